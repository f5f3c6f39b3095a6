"""The work that is timed when this library's speed is judged: SpecKV steps (score, select, compact), SpecPC keep
sets, the cascade of the two, and the selection with the gather alone, through the entry points of
paper_2506_08373_b200.binding, from one layer of a 2K prompt to all layers of a 128K one.

Inputs are seeded and made on the GPU.  Q, K and V are N(0,1) in bf16; the last feature of Q and K carries an additive
logit bias per key, -1.1 ln(rank) for a random ranking (approximately sparse attention), with a further drop of 2
behind the keys whose pooling windows just about fill the budget: the prompt has about as much that matters as the
caller keeps.  The drop also keeps neighbouring ranks apart where the budget cuts, so that correct implementations
with different rounding select the same positions and their lists can be compared."""
import math

import torch

from paper_2506_08373_b200 import binding as B

POOLS = {"max": B.POOL_MAX, "avg": B.POOL_AVG, "avg_then_max": B.POOL_AVG_THEN_MAX}
REDUCES = {"sum": B.REDUCE_SUM, "max": B.REDUCE_MAX}

LLAMA_8B = dict(layers=32, q_heads=32, kv_heads=8, dim=128)
LLAMA_1B_DRAFT = dict(layers=16, q_heads=32, kv_heads=8, dim=64)
# every case has all of these; what a kind does not use stays at its default
DEFAULTS = dict(layers=1, q_heads=32, kv_heads=8, dim=128, seqs=1, tokens=0, len_lo=0, len_hi=0, lookahead=64, window=32,
                pool="max", pool_k=7, budget=1024, vert=0, forced=0, reduce="sum", causal=0, weights=0, token_major=0,
                page=0, neighbor=0, skip=0)


def case(kind, **kw):
    c = dict(DEFAULTS, kind=kind)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: one layer of a short prompt, where launches and host time count
        case("kv", name="tiny_2k", q_heads=8, kv_heads=2, dim=64, tokens=2048, lookahead=32, window=16, budget=256),
        # sparse prefill goes layer by layer: one layer's scores, cache and vertical indices and compacted rows; odd
        # length, causal window, window always kept, K/V in the token-major layout that projections write
        case("kv", name="layer_12k", tokens=12345, vert=2048, forced=32, causal=1, token_major=1),
        # the same at a long prompt
        case("kv", name="layer_64k", tokens=65536, vert=2048, forced=32, budget=2048),
        # all layers of a 16K prompt: the ordinary step
        case("kv", name="step_16k", tokens=16384, **LLAMA_8B),
        # all layers of a 128K prompt with a longer lookahead: the largest step, and the benchmark's default
        case("kv", name="step_128k", tokens=131072, lookahead=128, budget=2048, **LLAMA_8B),
        # selection and gather alone on scores in hand (a cache cut again to another budget)
        case("select", name="select_gather_128k", tokens=131072, budget=2048, **LLAMA_8B),
        # no lookahead at all: the prompt's own window scores the keys (the SnapKV special case)
        case("kv", name="window_only_32k", tokens=32768, lookahead=0, window=32, forced=32, **LLAMA_8B),
        # the longest lookahead of the latency study (more query rows than stay resident at once), with the
        # max reduction and average pooling that Algorithm 1 prints
        case("kv", name="lookahead512_32k", layers=8, tokens=32768, lookahead=512, reduce="max", pool="avg"),
        # ragged batch into a paged cache; 8 of the model's 32 layers, so that three states fit the card
        case("kv", name="ragged_paged_16seq", layers=8, seqs=16, len_lo=4096, len_hi=65536, page=16),
        # SpecPC on a draft model: scores of all layers and heads to one keep list
        case("pc", name="specpc_32k", tokens=32768, lookahead=64, window=64, budget=4096, neighbor=8, **LLAMA_1B_DRAFT),
        # SpecPC with the hyper-parameter table's settings: one lookahead row, max reductions, window row weights,
        # average pool then max pool, the first layers left out, window always kept
        case("pc", name="specpc_paper_32k", tokens=32768, lookahead=1, window=64, budget=1024, neighbor=64, skip=8,
             pool="avg_then_max", pool_k=64, reduce="max", weights=1, forced=64, **LLAMA_1B_DRAFT),
        # SpecKV-PC: the draft's scores cut the prompt to 2048 tokens, their K/V rows are packed, and SpecKV runs on
        # the packed prompt, without the host in between
        case("cascade", name="cascade_32k", tokens=32768, budget=256, **LLAMA_8B),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def odd(n):                      # half of the lengths are as they come, half rounded as a user pads them
        return n if rng.random() < 0.5 else max(64, n // 64 * 64)

    kind = rng.choice(["kv", "kv", "kv", "kv", "pc", "pc", "select", "cascade"])
    tokens = odd(log_int(2048, 131072))
    if kind == "pc":
        paper = rng.random() < 0.5
        tokens = min(tokens, 65536)
        c = case(kind, layers=rng.choice([8, 12, 16, 24]), q_heads=32, kv_heads=8, dim=64, tokens=tokens,
                 lookahead=1 if paper else log_int(8, 128), window=rng.choice([32, 64]), budget=max(64, tokens // rng.choice([8, 16, 32])),
                 neighbor=64 if paper else rng.choice([4, 8]))
        if paper:
            c.update(pool="avg_then_max", pool_k=64, reduce="max", weights=1, forced=c["window"], skip=rng.choice([0, 4]))
    elif kind == "cascade":
        c = case(kind, layers=rng.choice([8, 16, 32]), tokens=min(tokens, 65536) + 2048, budget=rng.choice([128, 256, 512]),
                 lookahead=log_int(16, 128))
    else:
        group = rng.choice([1, 2, 4, 4, 4, 5, 8])
        kv_heads = rng.choice([2, 4, 8, 8, 8])
        c = case(kind, layers=rng.choice([1, 1, 2, 8, 16, 32]), q_heads=group * kv_heads, kv_heads=kv_heads,
                 dim=rng.choice([64, 128, 128]), tokens=tokens, lookahead=rng.choice([0, log_int(8, 160), log_int(8, 160), log_int(160, 512)]),
                 window=rng.choice([16, 32, 32, 48]), budget=rng.choice([256, 512, 1024, 2048]))
        c["budget"] = min(c["budget"], tokens // 8)
        if rng.random() < 0.3:
            c.update(vert=min(2048, tokens // 6))
        if rng.random() < 0.5:
            c.update(forced=min(c["window"], c["budget"] // 2), causal=1, token_major=rng.choice([0, 1]))
        if rng.random() < 0.25:
            c.update(reduce="max", pool="avg", pool_k=rng.choice([5, 7, 13]))
        if kind == "kv" and rng.random() < 0.3:
            seqs = rng.choice([2, 5, 16])
            c.update(seqs=seqs, len_lo=max(1024, tokens // 16), len_hi=max(2048, tokens), page=rng.choice([0, 16, 64]),
                     token_major=0)
            c["budget"] = min(c["budget"], c["len_lo"] // 4)
            c["vert"] = 0
    big = next(x for x in listed() if x["name"] == "step_128k")
    while c["layers"] > 1 and (_work_flops(c) > _work_flops(big) / 2 or _cache_bytes(c) > _cache_bytes(big)):
        c["layers"] = max(1, c["layers"] // 2)
        c["skip"] = min(c["skip"], c["layers"] - 1)
    while _work_flops(c) > _work_flops(big) / 2 or _cache_bytes(c) > _cache_bytes(big):
        c["lookahead"] = min(c["lookahead"] // 2, 64)
        if c["seqs"] > 1:
            c["seqs"] //= 2
    return c


# ------------------------------------------------------------------------- inputs ---------

def _lengths(c):
    """Prompt length of every sequence; a property of the case, so that all seeds have one shape."""
    if c["seqs"] == 1:
        return [c["tokens"] or c["len_hi"]]
    lo, hi, n = c["len_lo"], c["len_hi"], c["seqs"]
    return [lo + (hi - lo) * ((i * 7919 + 1237) % 1009) // 1009 for i in range(n)]      # spread over [lo, hi)


def _cache_bytes(c):
    return 4 * c["layers"] * c["kv_heads"] * sum(_lengths(c)) * c["dim"]


def _work_flops(c):
    return 2.0 * c["layers"] * c["q_heads"] * (c["lookahead"] + c["window"]) * sum(_lengths(c)) * c["dim"]


def _width(c):
    """How wide a single heavy key shows in the pooled scores."""
    return c["pool_k"] + c["neighbor"] - 1 if c["pool"] == "avg_then_max" else c["pool_k"]


def _knee(n, budget, width):
    """How many of n keys at random places have pooling windows (width wide) that cover about 0.97 of the budget."""
    return max(1, int(n * (1.0 - (1.0 - min(0.97 * budget / n, 0.9)) ** (1.0 / width))))


def _bias(gen, rows, lens, budget, width):
    """fp32 [rows, total] logit bias per key: -1.1 ln(rank), two less behind the knee."""
    out = []
    for n in lens:
        rank = torch.rand((rows, n), generator=gen, device="cuda").argsort(1).argsort(1).float().add_(1.0)
        out.append(rank.log().mul_(-1.1).sub_((rank > _knee(n, budget, width)).float().mul_(2.0)))
    return torch.cat(out, 1)


def _queries(gen, c, seqs, layers, dim, rows, scale):
    q = torch.randn((seqs, layers, c["q_heads"], rows, dim), generator=gen, device="cuda", dtype=torch.bfloat16)
    q[..., dim - 1] = 1.0 / scale
    return q


def _cache(gen, c, layers, dim, total, token_major=0):
    """[layers, kv_heads, total, dim] bf16, a view of a token-major array where the case says so."""
    H = c["kv_heads"]
    shape = (layers, total, H, dim) if token_major else (layers, H, total, dim)
    x = torch.empty(shape, device="cuda", dtype=torch.bfloat16)
    for l in range(layers):
        x[l].normal_(generator=gen)
    return x.transpose(1, 2) if token_major else x


def _problem(c, lens, layers, dim, cu, k=None, v=None, total=0, bound=0):
    return B.make_problem(n_layers=layers, n_q_heads=c["q_heads"], n_kv_heads=c["kv_heads"], head_dim=dim,
                          n_lookahead=c["lookahead"], n_window=c["window"], softmax_scale=1.0 / math.sqrt(dim),
                          total_tokens=total or sum(lens), n_in=bound or max(lens), n_seq=len(lens), cu_seqlens=cu, k=k, v=v)


def _workspace(pr):
    return torch.empty(max(B.spec_workspace_bytes(pr), 16), dtype=torch.uint8, device="cuda")


def _ints(*shape):
    return torch.empty(shape, dtype=torch.int32, device="cuda")


def prepare(c, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    lens = _lengths(c)
    total, L, H, d, S = sum(lens), c["layers"], c["kv_heads"], c["dim"], len(lens)
    st = {"case": c, "status": torch.zeros(1, dtype=torch.int32, device="cuda"), "cu": None, "weight": None}
    if S > 1:
        cu = [0]
        for n in lens:
            cu.append(cu[-1] + n)
        st["cu"] = torch.tensor(cu, dtype=torch.int32, device="cuda")
    if c["kind"] in ("pc", "cascade"):
        draft = c if c["kind"] == "pc" else _draft_of(c)
        st["draft"] = _prepare_pc(gen, draft, lens, st)
    if c["kind"] == "pc":
        return st
    st["k"] = _cache(gen, c, L, d, total, c["token_major"])
    st["v"] = _cache(gen, c, L, d, total, c["token_major"])
    if c["kind"] == "cascade":
        p = st["draft"]
        cap = p["cap"]
        st["pr"] = _problem(c, lens, L, d, None, st["k"], st["v"])
        st["k_kept"] = torch.empty((L, H, cap, d), device="cuda", dtype=torch.bfloat16)
        st["v_kept"] = torch.empty_like(st["k_kept"])
        st["cu_kept"] = _ints(2)
        for l in range(L):
            st["k"][l, :, :, d - 1] = _bias(gen, H, lens, c["budget"] * lens[0] // cap, _width(c))
        st["pr_kept"] = _problem(c, [cap], L, d, st["cu_kept"], st["k_kept"], st["v_kept"])
        pr_step = st["pr_kept"]
    else:
        pr_step = st["pr"] = _problem(c, lens, L, d, st["cu"], st["k"], st["v"])
    st["ws"] = _workspace(pr_step)
    n_scored = pr_step.total_tokens
    if c["kind"] == "select":
        # scores as the scoring step leaves them: per head, the rows' softmax weights summed over the group
        rows = (c["q_heads"] // H) * (c["lookahead"] + c["window"])
        st["scores"] = torch.empty((L, H, total), dtype=torch.float32, device="cuda")
        for l in range(L):
            s = _bias(gen, H, lens, c["budget"], _width(c)).add_(torch.randn((H, total), generator=gen, device="cuda").mul_(0.1)).exp_()
            st["scores"][l] = s * (rows / s.sum(1, keepdim=True))
    else:
        st["q"] = _queries(gen, c, S, L, d, c["lookahead"] + c["window"], 1.0 / math.sqrt(d))
        if c["kind"] == "kv":
            for l in range(L):
                st["k"][l, :, :, d - 1] = _bias(gen, H, lens, c["budget"], _width(c))
        st["scores"] = torch.empty((L, H, n_scored), dtype=torch.float32, device="cuda")
    C = c["budget"]
    st["idx"], st["cnt"] = _ints(S, L, H, C), _ints(S, L, H)
    if c["vert"]:
        st["vidx"], st["vcnt"] = _ints(S, L, H, c["vert"]), _ints(S, L, H)
    if c["page"]:
        pages = (C + c["page"] - 1) // c["page"]
        st["pages"] = S * pages
        st["table"] = torch.randperm(S * pages, generator=gen, device="cuda").to(torch.int32).view(S, pages)
        shape = (L, S * pages, H, c["page"], d)
        st["k_out"] = torch.zeros(shape, device="cuda", dtype=torch.bfloat16)
        st["v_out"] = torch.zeros(shape, device="cuda", dtype=torch.bfloat16)
    else:
        st["k_out"] = torch.empty((S, L, H, C, d), device="cuda", dtype=torch.bfloat16)
        st["v_out"] = torch.empty_like(st["k_out"])
    return st


def _draft_of(c):
    """The draft pass of a cascade: 2048 tokens kept, with the hyper-parameter table's pooling."""
    return case("pc", tokens=c["tokens"], layers=16, q_heads=c["q_heads"], kv_heads=c["kv_heads"], dim=64, lookahead=1, window=32,
                budget=2016, neighbor=64, pool="avg_then_max", pool_k=64, reduce="max", weights=1, forced=32, skip=8)


def _prepare_pc(gen, c, lens, st):
    """A draft model's Q and K; what matters is a property of the token, the same in all layers and heads."""
    L, H, d, n = c["layers"], c["kv_heads"], c["dim"], lens[0]
    p = {"case": c}
    p["k"] = _cache(gen, c, L, d, n)
    p["k"][..., d - 1] = _bias(gen, 1, lens, c["budget"], _width(c))[0]
    p["q"] = _queries(gen, c, 1, L, d, c["lookahead"] + c["window"], 1.0 / math.sqrt(d))
    p["pr"] = _problem(c, lens, L, d, None, p["k"])
    p["pr_keep"] = _problem(c, lens, L - c["skip"], d, None)
    p["ws"] = _workspace(p["pr"])
    p["scores"] = torch.empty((L, H, n), dtype=torch.float32, device="cuda")
    if c["weights"]:                 # window row j of w weighs j / w, lookahead rows 1
        p["weight"] = torch.cat([torch.arange(1, c["window"] + 1, device="cuda").float() / c["window"],
                                 torch.ones(c["lookahead"], device="cuda")])
    widest = c["budget"] if c["pool"] == "avg_then_max" else c["budget"] * (2 * c["neighbor"] + 1)
    p["cap"] = min(n, widest + c["forced"])
    p["keep"], p["n_keep"] = _ints(1, p["cap"]), _ints(1)
    return p


# -------------------------------------------------------------------------- a pass --------

def _run_pc(p, status):
    c = p["case"]
    B.spec_score(p["pr"], p["q"], p["k"], p["scores"], p["ws"], row_weight=p.get("weight"), reduce=REDUCES[c["reduce"]],
                 status_word=status)
    B.specpc_token_select(p["pr_keep"], p["scores"][c["skip"]:], REDUCES[c["reduce"]], POOLS[c["pool"]], c["pool_k"], c["budget"],
                          c["neighbor"], c["forced"], p["keep"], p["cap"], p["n_keep"], p["ws"], status_word=status)


def run(st):
    c, status = st["case"], st["status"]
    if c["kind"] in ("pc", "cascade"):
        p = st["draft"]
        _run_pc(p, status)
        out = {"draft_scores": p["scores"], "keep": p["keep"], "n_keep": p["n_keep"]}
        if c["kind"] == "pc":
            return out
        B.spec_gather_tokens(st["pr"], st["k"], st["v"], p["keep"], p["cap"], p["n_keep"], st["k_kept"], st["v_kept"], p["cap"],
                             st["cu_kept"], status_word=status)
        pr, k, v = st["pr_kept"], st["k_kept"], st["v_kept"]
        out.update(cu_kept=st["cu_kept"], k_kept=_bits(k), v_kept=_bits(v))
    else:
        pr, k, v, out = st["pr"], st["k"], st["v"], {}
    if c["kind"] != "select":
        B.spec_score(pr, st["q"], k, st["scores"], st["ws"], reduce=REDUCES[c["reduce"]], causal_window=c["causal"], status_word=status)
        out["scores"] = st["scores"]
    if c["vert"]:
        B.spec_pool_topk_vert(pr, st["scores"], POOLS[c["pool"]], c["pool_k"], c["budget"], c["forced"], st["idx"], st["cnt"], c["vert"],
                              st["vidx"], st["vcnt"], workspace=st["ws"], status_word=status)
        out.update(vidx=st["vidx"], vcnt=st["vcnt"])
    else:
        B.spec_pool_topk(pr, st["scores"], POOLS[c["pool"]], c["pool_k"], c["budget"], c["forced"], st["idx"], st["cnt"],
                         workspace=st["ws"], status_word=status)
    if c["page"]:
        B.spec_compact_kv(pr, k, v, st["idx"], c["budget"], st["k_out"], st["v_out"], block_table=st["table"], page_size=c["page"],
                          n_pages=st["pages"], status_word=status)
    else:
        B.spec_compact_kv(pr, k, v, st["idx"], c["budget"], st["k_out"], st["v_out"], status_word=status)
    out.update(idx=st["idx"], cnt=st["cnt"], k_out=_bits(st["k_out"]), v_out=_bits(st["v_out"]), status=status)
    return out


def _bits(x):
    """Gathered rows as whole values: they are copied bit for bit."""
    return x.view(torch.int16)


# -------------------------------------------------------------------------- its work ------

def work(c):
    """One contraction of the query rows with the keys; Q, K and the rows gathered read once, every output written once."""
    if c["kind"] == "cascade":
        d, kept = _draft_of(c), 2048
        w = work(d)
        on_kept = work(dict(c, kind="kv", tokens=kept))
        moved = 2 * _cache_bytes(dict(c, tokens=kept))
        return {"bytes": w["bytes"] + moved + on_kept["bytes"], "flops": w["flops"] + on_kept["flops"]}
    lens = _lengths(c)
    L, H, d, total, units = c["layers"], c["kv_heads"], c["dim"], sum(lens), len(lens) * c["layers"] * c["kv_heads"]
    b, flops = 4.0 * L * H * total, 0.0                                                 # the scores, written (or read) once
    if c["kind"] != "select":
        b += _cache_bytes(c) / 2 + 2.0 * len(lens) * L * c["q_heads"] * (c["lookahead"] + c["window"]) * d
        flops = _work_flops(c)
    if c["kind"] == "pc":
        return {"bytes": b + 4.0 * c["budget"], "flops": flops}
    return {"bytes": b + units * (4.0 * (c["budget"] + c["vert"]) + 8.0 * c["budget"] * d), "flops": flops}


def tolerance(c):
    """Against the same sums in 64 bits the scores are off by up to 5e-5 in the 2-norm and 1.1e-4 at worst (the max
    reduction, one exponential per score): four times that.  With scores off by 1e-5 each at random, up to 0.25 % of the
    index entries move (one list in a hundred shifts); whole values allow for a few times that."""
    return {"rel": 2e-4, "max": 5e-4, "differ": 0.01}
