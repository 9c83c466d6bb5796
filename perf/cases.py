"""What the speed of this library is measured on: the decode step, the dense decode, the summary build and the chunked
prefill, called through the binding as a serving program calls them.

Kinds of case
  step     a short generation: `steps` calls of CompKV.step, one token per sequence each (append, select, attend).  The
           scheduler hands over the sequences' lengths first, so that the same state can be run again.
  layers   one token through a stack of layers, each with its own cache, captured once as a CUDA graph and replayed (how
           a model runs the step).
  host     one step from pinned host buffers on a stream of the caller's own (CompKV.step_host).
  dense    dense decode attention over the whole cache (the fallback for layers that are not sparsified, and the baseline).
  build    summaries of a cache that somebody else filled (CompKV.stats_build).
  prefill  prompt chunks written to their pages with their summaries (CompKV.prefill).

Values follow the block mixture of paper_2609_26300_b200.synth (a centre per 16 tokens plus noise of 0.05, 0.3 or 1.0,
four outlier channels times eight, needles aligned with the query), drawn on the GPU.
"""
import math
import random

import torch

from paper_2609_26300_b200 import binding

PAGE, D = 16, 128
NEEDLES = 64


def _case(name, kind, batch, q_heads, kv_heads, ctx, **kw):
    case = {"name": name, "kind": kind, "batch": batch, "q_heads": q_heads, "kv_heads": kv_heads, "ctx": ctx,
            "ctx_min": ctx, "budget": 2048, "block": 16, "r": 4, "stat_bf16": 0, "steps": 16, "layers": 1, "chunk": 0}
    case.update(kw)
    return case


def listed():
    return [
        # the smallest call: one KV head, a short cache (synth.CONFIGS[1]); launches and latency are all there is
        _case("step_4k_b1_one_head", "step", 1, 4, 1, 4096, budget=256),
        # one user, an 8B-class layer, a medium prompt (synth.CONFIGS[2])
        _case("step_32k_b1", "step", 1, 32, 8, 32768, budget=1024),
        # four users at the full context (synth.CONFIGS[3], the benchmark's workload)
        _case("step_128k_b4", "step", 4, 32, 8, 131072),
        # a continuous batch with ragged lengths and groups of eight (synth.CONFIGS[4])
        _case("step_ragged_b16_group8", "step", 16, 64, 8, 65536, ctx_min=16384, budget=1024),
        # one user at the full context, longer blocks and the largest budget (a point of the synth.CONFIGS[5] sweep)
        _case("step_128k_b1_block32", "step", 1, 32, 8, 131072, budget=4096, block=32),
        # the compact summary layout, lengths that fill neither block nor page
        _case("step_bf16_summaries_b3", "step", 3, 32, 8, 100003, ctx_min=60001, stat_bf16=1),
        # a variance per coordinate (the method's other operating point)
        _case("step_r128_b2", "step", 2, 32, 8, 90001, r=128),
        # a model's loop: one token through eight layers, one graph replay
        _case("layers8_64k_b1_graph", "layers", 1, 32, 8, 65536, layers=8, budget=1024, steps=1),
        # a caller whose activations live on the host: pinned buffers in and out, one step per call
        _case("host_step_128k_b1", "host", 1, 32, 8, 131072, steps=1),
        # dense decode over the benchmark's cache
        _case("dense_128k_b4", "dense", 4, 32, 8, 131072, steps=1),
        # summaries of a prefilled 128K cache, one sequence (part of the synth.CONFIGS[5] sweep)
        _case("build_128k_b1", "build", 1, 32, 8, 131072, steps=1),
        # a 32K prompt in four chunks, two sequences
        _case("prefill_32k_b2_chunks", "prefill", 2, 32, 8, 32768, chunk=8192, steps=1),
    ]


def draw(rng):
    def logu(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["step"] * 6 + ["layers", "host", "dense", "dense", "build", "prefill"])
    q_heads, kv_heads = rng.choice([(32, 8), (32, 8), (64, 8), (16, 8), (8, 8), (4, 1)])
    batch = logu(1, 16)
    ctx = min(logu(2000, 131072), 4 * 131072 // batch)
    if rng.random() < 0.3:
        ctx = max(1024, ctx // 1024 * 1024)
    ctx_min = ctx if rng.random() < 0.5 else max(500, int(ctx * rng.uniform(0.25, 1.0)))
    block = rng.choice([16, 16, 16, 32, 64])
    budget = rng.choice([512, 1024, 2048, 4096])
    budget = budget if budget <= ctx else 512
    r = rng.choice([4] * 5 + [128, 16, 1])
    stat_bf16 = int(r < D and rng.random() < 0.2)
    kw = {"ctx_min": ctx_min, "block": block, "budget": budget, "r": r, "stat_bf16": stat_bf16}
    if kind != "step":
        kw["steps"] = 1
    if kind == "layers":
        batch = min(batch, 2)
        ctx = min(ctx, 65536)
        kw.update(layers=rng.choice([2, 4, 8]), ctx_min=min(ctx_min, ctx))
    if kind == "prefill":
        ctx = min(ctx, 65536)
        kw.update(ctx_min=min(ctx_min, ctx), chunk=min(ctx, logu(512, 16384)))
    case = _case("", kind, batch, q_heads, kv_heads, ctx, **kw)
    del case["name"]
    most = max(work(c)["bytes"] for c in listed())
    while work(case)["bytes"] > most:   # no more work than the largest listed case
        case["ctx"] = case["ctx"] * 4 // 5
        case["ctx_min"] = min(case["ctx_min"], case["ctx"])
    return case


def _lens(case):
    """Tokens per sequence before the pass: part of the case, the same for every seed."""
    rng = random.Random("%(batch)d %(ctx)d %(ctx_min)d" % case)
    return [case["ctx"] if i == 0 else rng.randint(case["ctx_min"], case["ctx"]) for i in range(case["batch"])]


class _Layer:
    """One layer's cache as a serving program holds it: pools, page table, lengths, context; and its queries and new rows."""

    def __init__(self, case, gen, lens):
        dev = torch.device("cuda")
        b, hq, hkv, steps = case["batch"], case["q_heads"], case["kv_heads"], case["steps"]
        self.lens0 = torch.tensor(lens, dtype=torch.int32, device=dev)
        self.lens = self.lens0.clone()
        self.max_len = max(lens) + steps                      # what the host knows: an upper bound for the whole pass
        cap = (self.max_len + 1023) // 1024 * 1024            # page-table rows are sized in units of 1024 tokens
        need = [-(-(n + steps) // PAGE) for n in lens]
        self.num_pages = sum(need)
        order = torch.randperm(self.num_pages, generator=gen, device=dev, dtype=torch.int32)
        self.table = torch.full((b, cap // PAGE), -1, dtype=torch.int32, device=dev)
        at = 0
        for s, n in enumerate(need):
            self.table[s, :n] = order[at:at + n]
            at += n
        dt = torch.bfloat16

        def normal(*shape):
            return torch.randn(*shape, generator=gen, device=dev, dtype=dt)

        scale = torch.ones(hkv, 1, D, device=dev, dtype=dt)
        channels = torch.rand(hkv, D, generator=gen, device=dev).argsort(1)[:, :4]
        scale.view(hkv, D).scatter_(1, channels, 8.0)
        levels = torch.tensor([0.05, 0.3, 1.0], device=dev, dtype=dt)

        def mixture(rows, per):   # [rows][per][hkv? ...] key rows around a centre
            k = normal(rows, hkv, per, D)
            k.mul_(levels[torch.randint(0, 3, (rows, hkv, 1, 1), generator=gen, device=dev)])
            return k.add_(normal(rows, hkv, 1, D)).mul_(scale)

        self.k_pool, self.v_pool = mixture(self.num_pages, PAGE), normal(self.num_pages, hkv, PAGE, D)
        self.q = normal(1, b, hq, D) + 0.3 * normal(steps, b, hq, D)
        # the rows of the steps continue the mixture: one centre per sequence
        self.k_new = mixture(b, steps).permute(2, 0, 1, 3).contiguous()
        self.v_new = normal(steps, b, hkv, D)
        # needles: tokens whose keys lean towards the group's mean query by six units of logit
        qbar = self.q[0].view(b, hkv, hq // hkv, D).float().mean(2)
        bump = (6.0 * math.sqrt(D) / qbar.square().sum(-1, keepdim=True) * qbar).to(dt)
        heads = torch.arange(hkv, device=dev).view(hkv, 1)
        for s, n in enumerate(lens):
            pos = torch.randint(min(case["block"], n - 1), n, (hkv, min(NEEDLES, max(1, n // 64))), generator=gen, device=dev)
            self.k_pool[self.table[s][pos // PAGE].long(), heads, pos % PAGE] += bump[s][:, None, :]
        self.budget = case["budget"]
        self.ckv = binding.CompKV(hq, hkv, b, cap // case["block"], self.num_pages, block_size=case["block"],
                                  var_groups=case["r"], stat_bf16=case["stat_bf16"])
        self.steps = steps
        ko, do, vo = binding.stats_offsets(self.ckv.layout)
        rows = b * hkv * (cap // case["block"])
        mean = rows * D * (2 if case["stat_bf16"] else 4)
        st = self.ckv.stats
        self.summaries = [st[ko:ko + mean].view(dt), st[vo:vo + mean].view(dt)]
        self.summaries.append(st[do:do + rows * case["r"] * 4].view(dt if case["r"] == D else torch.float32))

    def outputs(self, steps):
        """Output buffers of `steps` steps, stacked, and the tuple each step writes."""
        one = self.ckv.alloc_outputs(self.lens.shape[0], self.budget)
        stacked = [torch.zeros((steps,) + tuple(t.shape), dtype=t.dtype, device=t.device) for t in one]
        return stacked, [tuple(t[i] for t in stacked) for i in range(steps)]


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    lens = _lens(case)
    kind = case["kind"]
    layers = [_Layer(case, gen, lens) for _ in range(case["layers"])]
    state = {"kind": kind, "layers": layers}
    L = layers[0]
    if kind in ("step", "layers", "host"):   # the summaries of the prompt exist when generation starts
        for x in layers:
            x.ckv.stats_build(x.k_pool, x.v_pool, x.table, x.lens, max(lens))
    if kind == "step":
        L.stacked, L.outs = L.outputs(L.steps)
        L.q_t, L.k_t, L.v_t = list(L.q), list(L.k_new), list(L.v_new)
    elif kind == "layers":
        lens_all = torch.stack([x.lens for x in layers])     # all layers' lengths in one array, set by one copy per token
        state["lens_all"], state["lens0_all"] = lens_all, lens_all.clone()

        def token():
            for x, n in zip(layers, lens_all):
                x.ckv.step(x.q[0], x.k_new[0], x.v_new[0], x.k_pool, x.v_pool, x.table, n, x.max_len, x.budget, x.outs[0])

        for x in layers:
            x.stacked, x.outs = x.outputs(1)
        token()
        torch.cuda.synchronize()
        state["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(state["graph"]):
            token()
    elif kind == "host":
        pin = {"dtype": torch.bfloat16, "pin_memory": True}
        b, hq, hkv = case["batch"], case["q_heads"], case["kv_heads"]
        L.hq, L.hk, L.hv = (torch.empty(*x.shape[1:], **pin).copy_(x[0]) for x in (L.q, L.k_new, L.v_new))
        L.ho = torch.zeros(b, hq, D, **pin)
        L.hi = torch.zeros(b, hkv, case["budget"] // case["block"], dtype=torch.int32, pin_memory=True)
        L.hc = torch.zeros(b, hkv, dtype=torch.int32, pin_memory=True)
        state["stream"] = torch.cuda.Stream()
        torch.cuda.synchronize()
    elif kind == "dense":
        L.out = torch.zeros(case["batch"], case["q_heads"], D, dtype=torch.bfloat16, device="cuda")
        L.lse = torch.zeros(case["batch"], case["q_heads"], device="cuda")
    elif kind == "prefill":
        # the prompt as the projections leave it: token-major rows, chunk after chunk; the pools start out empty
        n, c = case["ctx"], case["chunk"]
        pages = L.table[:, :-(-n // PAGE)].clamp_min(0).long()

        def rows(pool):
            x = pool[pages].permute(0, 1, 3, 2, 4).reshape(case["batch"], -1, case["kv_heads"], D)
            return [x[:, i:min(i + c, n)].contiguous() for i in range(0, n, c)]

        L.k_chunks, L.v_chunks = rows(L.k_pool), rows(L.v_pool)
        L.k_pool.zero_()
        L.v_pool.zero_()
        L.empty = torch.zeros_like(L.lens)
        L.new = [(L.lens0 - i).clamp(0, min(c, n - i)).to(torch.int32) for i in range(0, n, c)]
    return state


def run(state):
    kind, L = state["kind"], state["layers"][0]
    if kind == "step":
        L.lens.copy_(L.lens0)
        for t in range(L.steps):
            L.ckv.step(L.q_t[t], L.k_t[t], L.v_t[t], L.k_pool, L.v_pool, L.table, L.lens, L.max_len, L.budget, L.outs[t])
        return L.stacked + [L.lens] + L.summaries
    if kind == "layers":
        state["lens_all"].copy_(state["lens0_all"])
        state["graph"].replay()
        return [x.stacked + x.summaries for x in state["layers"]] + [state["lens_all"]]
    if kind == "host":
        with torch.cuda.stream(state["stream"]):
            L.lens.copy_(L.lens0)
            L.ckv.step_host(L.hq, L.hk, L.hv, L.k_pool, L.v_pool, L.table, L.lens, L.max_len, L.budget, L.ho, L.hi, L.hc)
        return [L.ho, L.hi, L.hc, L.lens] + L.summaries
    if kind == "dense":
        L.ckv.dense_decode(L.q[0], L.k_pool, L.v_pool, L.table, L.lens, L.max_len, L.out, L.lse)
        return [L.out, L.lse]
    if kind == "build":
        L.ckv.stats_build(L.k_pool, L.v_pool, L.table, L.lens, L.max_len)
        return L.summaries
    L.lens.copy_(L.empty)
    for k, v, n in zip(L.k_chunks, L.v_chunks, L.new):
        L.ckv.prefill(L.k_pool, L.v_pool, L.table, L.lens, k, v, n, k.shape[1])
    return L.summaries + [L.k_pool, L.v_pool, L.lens]


def work(case):
    """Bytes and operations of one pass: summaries as the step reads them (mean keys in full, mean values at bf16 with the
    default layout), the selected tokens' keys and values, new rows, queries and results."""
    hq, hkv, bs, r = case["q_heads"], case["kv_heads"], case["block"], case["r"]
    g, kind, lens = hq // hkv, case["kind"], _lens(case)
    mean = 2 * D if case["stat_bf16"] else 4 * D
    total = flops = 0
    if kind in ("step", "layers", "host"):
        for t in range(1, case["steps"] + 1):
            for n in lens:
                x = -(-(n + t) // bs)
                sel = min(case["budget"], n + t)
                row = mean + (2 * D if r == 4 else mean) + 4 * r
                total += hkv * (x * row + sel * 4 * D + 4 * D + 2 * g * 2 * D)
                flops += hkv * g * (x * (4 * D + 2 * r) + sel * 4 * D)
        total, flops = total * case["layers"], flops * case["layers"]
    elif kind == "dense":
        total = sum(hkv * (n * 4 * D + 2 * g * 2 * D) for n in lens)
        flops = sum(hq * n * 4 * D for n in lens)
    else:
        passes = 2 if kind == "prefill" else 1   # a prefill reads the rows and writes the pages
        total = sum(hkv * (passes * n * 4 * D + -(-n // bs) * (2 * mean + 4 * r)) for n in lens)
        flops = sum(hkv * n * 5 * D for n in lens)
    return {"bytes": total, "flops": flops}


def tolerance(case):
    # Outputs are rounded once to bf16: against a 64-bit evaluation the dense pass shows a relative error of 1.7e-3 and a
    # largest one of 3.7e-3.  Ids may differ where two scores tie to fp32 rounding.  Summaries are fp32 sums of 16 to 64
    # rows stored as bf16 pairs: a mean on a rounding boundary moves its hi half by an ulp and its lo half by as much the
    # other way, 1.8e-5 relative and 0.025 at most against 64-bit sums; rows of the cache come back unchanged.
    if case["kind"] in ("step", "layers", "host"):
        return {"rel": 7e-3, "max": 0.1, "differ": 5e-3}
    if case["kind"] == "dense":
        return {"rel": 7e-3, "max": 0.02}
    return {"rel": 8e-5, "max": 0.1}
