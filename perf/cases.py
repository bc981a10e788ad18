"""Workloads of the tail-replay library, timed through its public Python entry points.

A case is a dict of plain values.  ``kind`` says which call a serving program makes:

    replay   one ``gdn_tail_replay`` over a batch of prefix-cache hits (one layer)
    rebuild  the same call once per linear-attention layer, back to back, for one hit
    prefill  ``gdn_full_prefill`` over a whole prefix
    decode   ``gdn_decode_step``: one token per request from the states of the replay

The other keys are the sizes (requests, tail lengths lo..hi, heads, head dims) and the options of the call: io dtype
(``bf16``/``f32``), ``raw`` (fused input stage), ``resume`` (start from a given state) and ``host`` (host-memory call).
Values follow the library's input recipe: unit keys and queries, v ~ N(0,1), log-decay ~ U(-0.1, -0.001),
beta = sigmoid(N(0,1)); raw inputs carry un-normalised q, k and the two pre-activations.
"""
import math
import random

import torch

import paper_2608_30310_b200 as gdn


def _case(kind, name=None, **kw):
    c = {"kind": kind, "requests": 1, "lo": 64, "hi": 64, "layers": 1, "hq": 16, "hv": 32, "dk": 128, "dv": 128,
         "io": "bf16", "raw": False, "resume": False, "host": False}
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one user continuing after the replay: the latency of a single token at the hybrid-model head shape
        _case("decode", "decode_1_request"),
        # a full serving batch, one token each: 1 GiB of states read and written
        _case("decode", "decode_256_requests", requests=256),
        # the smallest named configuration: fp32, d = 64, 4 heads, 512 tokens
        _case("replay", "tiny_fp32", lo=512, hi=512, hq=4, hv=4, dk=64, dv=64, io="f32"),
        # fp32 inputs at the hybrid-model shape: a few ragged hits
        _case("replay", "fp32_4_hits", requests=4, lo=401, hi=1639, io="f32"),
        # one layer of one hit: 5 % of a 32K prefix
        _case("replay", "single_layer_1638", lo=1638, hi=1638),
        # the whole state rebuild of one hit, 36 layers one after the other: 5 % of an 8K prefix
        _case("rebuild", "rebuild_8k_5pct_36_layers", lo=410, hi=410, layers=36),
        # a handful of hits at 10 % of 32K, ragged
        _case("replay", "hits_4_ragged_long", requests=4, lo=3121, hi=3277),
        # the headline batch: 32 concurrent hits with ragged tails
        _case("replay", "concurrent_32_hits", requests=32, lo=400, hi=3300),
        # projection outputs in, the input stage fused into the replay
        _case("replay", "raw_8_hits", requests=8, lo=410, hi=3277, raw=True),
        # suffixes served from the states of an earlier request: short, ragged, non-zero start
        _case("replay", "resume_16_suffixes", requests=16, lo=33, hi=700, resume=True),
        # the comparison the replay replaces: the whole 32K prefix of one request
        _case("prefill", "full_prefill_32k", lo=32768, hi=32768),
        # inputs and results in pinned host memory, staged by the library
        _case("replay", "host_memory_8_hits", requests=8, lo=410, hi=1639, host=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["replay", "rebuild", "prefill", "decode"], [6, 1, 1, 2])[0]
    if kind == "decode":
        return _case("decode", requests=_log_int(rng, 1, 256), io=rng.choice(["bf16", "bf16", "f32"]))
    if kind == "prefill":
        n = _log_int(rng, 4000, 32768)
        return _case("prefill", lo=n, hi=n)
    if kind == "rebuild":
        n = _log_int(rng, 200, 1200)
        return _case("rebuild", lo=n, hi=n, layers=rng.choice([12, 24, 36]))
    if rng.random() < 0.25:                        # fp32: every head shape, bounded by the listed fp32 work
        dk, dv = rng.choice([64, 128]), rng.choice([64, 128])
        hq, hv = rng.choice([(4, 4), (16, 32), (8, 16)])
        hi = _log_int(rng, 100, 1639)
        return _case("replay", requests=rng.randint(1, 4), lo=max(1, hi // rng.randint(1, 4)), hi=hi, hq=hq, hv=hv,
                     dk=dk, dv=dv, io="f32", raw=rng.random() < 0.2)
    hq, hv = rng.choice([(16, 32), (16, 32), (16, 16), (8, 32)])
    hi = _log_int(rng, 65, 3300)
    c = _case("replay", requests=_log_int(rng, 1, 32), lo=max(1, hi // rng.randint(1, 8)), hi=hi, hq=hq, hv=hv,
              raw=rng.random() < 0.2, resume=rng.random() < 0.25, host=rng.random() < 0.1)
    c["requests"] = max(1, min(c["requests"], 100000 // (c["lo"] + c["hi"])))     # no more tokens than the listed batch
    if c["host"]:                                  # the link into the device bounds these: keep them to the listed size
        c["requests"], c["hi"] = min(c["requests"], 8), min(c["hi"], 1639)
        c["lo"] = min(c["lo"], c["hi"])
    return c


def _tails(case):
    """Tail lengths of the batch: fixed by the sizes of the case, so that work() and prepare() agree."""
    r = random.Random("%d/%d/%d" % (case["requests"], case["lo"], case["hi"]))
    return [r.randint(case["lo"], case["hi"]) for _ in range(case["requests"])]


def _inputs(gen, dev, T, c, raw):
    dt = torch.bfloat16 if c["io"] == "bf16" else torch.float32

    def normal(*shape):
        return torch.randn(shape, generator=gen, device=dev, dtype=torch.float32)

    def uniform(lo, hi, *shape):
        return torch.rand(shape, generator=gen, device=dev, dtype=torch.float32) * (hi - lo) + lo

    q, k = normal(T, c["hq"], c["dk"]), normal(T, c["hq"], c["dk"])
    if raw:
        q, k = q * uniform(0.5, 3.0, T, c["hq"], 1), k * uniform(0.5, 3.0, T, c["hq"], 1)
        g, beta = uniform(2.2, 7.0, T, c["hv"]), normal(T, c["hv"])
    else:
        q, k = torch.nn.functional.normalize(q, dim=-1), torch.nn.functional.normalize(k, dim=-1)
        g, beta = uniform(-0.1, -0.001, T, c["hv"]), torch.sigmoid(normal(T, c["hv"]))
    v = normal(T, c["hv"], c["dv"])
    return q.to(dt), k.to(dt), v.to(dt), g, beta


def prepare(case, seed):
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    N, Hv, dk, dv = case["requests"], case["hv"], case["dk"], case["dv"]
    s = {"kind": case["kind"]}
    if case["kind"] == "decode":
        s["in"] = _inputs(gen, dev, N, case, False)
        s["state_in"] = torch.randn((N, Hv, dk, dv), generator=gen, device=dev)
        s["state_out"] = torch.empty_like(s["state_in"])
        s["o"] = torch.empty_like(s["in"][2])
        return s

    tails = _tails(case)
    cu = [0]
    for t in tails:
        cu.append(cu[-1] + t)
    T, L = cu[-1], case["layers"]
    cu = torch.tensor(cu, dtype=torch.int32, device=dev)
    init = torch.randn((N, Hv, dk, dv), generator=gen, device=dev) if case["resume"] else None
    ins = [_inputs(gen, dev, T, case, case["raw"]) for _ in range(L)]
    if case["host"]:
        cu, init = cu.cpu().pin_memory(), None if init is None else init.cpu().pin_memory()
        ins = [tuple(x.cpu().pin_memory() for x in xs) for xs in ins]
    where = {"pin_memory": True} if case["host"] else {"device": dev}
    s["o"] = torch.empty((L, T, Hv, dv), dtype=ins[0][2].dtype, **where)
    s["state"] = torch.empty((L, N, Hv, dk, dv), dtype=torch.float32, **where)
    s["workspace"] = gdn.Workspace(device=dev)
    s["options"] = {"raw_inputs": case["raw"], "init_state": init}
    s["layers"] = [(q, k, v, g, beta, cu, 64, s["o"][i], s["state"][i]) for i, (q, k, v, g, beta) in enumerate(ins)]
    return s


def run(s):
    if s["kind"] == "decode":
        q, k, v, g, beta = s["in"]
        gdn.gdn_decode_step(q, k, v, g, beta, s["state_in"], s["o"], s["state_out"])
        return s["o"], s["state_out"]
    call = gdn.gdn_full_prefill if s["kind"] == "prefill" else gdn.gdn_tail_replay
    for args in s["layers"]:
        call(*args, workspace=s["workspace"], **s["options"])
    return s["o"], s["state"]


def work(case):
    N, hq, hv, dk, dv = case["requests"], case["hq"], case["hv"], case["dk"], case["dv"]
    e = 2 if case["io"] == "bf16" else 4
    state = N * hv * dk * dv * 4
    T = N if case["kind"] == "decode" else sum(_tails(case))
    given = case["kind"] == "decode" or case["resume"]
    # q, k, v, o in the io dtype, log-decay and beta in fp32; the states written once, and read once where given;
    # per token and head S k, the rank-1 update and S q
    once = T * (2 * hq * dk * e + 2 * hv * dv * e + 2 * hv * 4) + state * (2 if given else 1)
    return {"bytes": case["layers"] * once, "flops": case["layers"] * 6.0 * dk * dv * T * hv}


def tolerance(case):
    if case["io"] == "f32":
        return {"rel": 1e-5}                       # fp32 throughout
    if case["kind"] == "decode":
        return {"rel": 2e-3}                       # fp32 arithmetic on bf16 inputs, one rounding of the output to bf16
    return {"rel": 1e-2}                           # bf16 operands of the chunk products, fp32 accumulation and state
