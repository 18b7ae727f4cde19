"""The measured cases: what programs that use the controller have it do, through its public entry points.

A case is one pass of such a program on inputs made from a seed:

- ``step``        one ``Session.step`` call (the first decision of a short chat turn), issued eagerly;
- ``plan``        one fused iteration through a recorded host-staged plan: hidden states from pinned host
                  memory, verification + step, the decisions back in host memory;
- ``decode``      T fused greedy iterations (``switchsd_verify_step``) of G batches, recorded once as a CUDA
                  graph and replayed, as a serving loop records its launch-bound part; G > 1 batches take
                  turns (micro-batches), which allows the prefetch of contexts and hidden states;
- ``sampled``     the same at T > 0 (``switchsd_verify_sampled_step``), the probe reading row a_b of the
                  target's [B, k+1, d] output;
- ``candidates``  the same with W candidates of D tokens (``switchsd_verify_candidates_step``);
- ``mlp``         the same as decode with the two-layer probe;
- ``index``       the same as decode with the incremental n-gram index instead of the rescan;
- ``index_build`` the index of a batch of prompts built, then the first step on it (prefill);
- ``labels``      the copy-mode labels of every position of a batch (training the probe).

The text is Zipf(1.1) prose or uniform ids with planted copies of earlier spans, or code (blocks tiled with
edits); half of the rows end inside a copy.  The target's tokens follow a stream per row (the copy's
continuation with edits, or the text's own law), drafts agree with it with probability 0.75 a token.
"""
import ctypes
import math

import torch

from paper_2609_20186_gb300 import Session
from paper_2609_20186_gb300 import binding as bd

GRAPHED = ("decode", "sampled", "candidates", "mlp", "index")


def _case(name, kind, B, L, **kw):
    c = dict(name=name, kind=kind, B=B, L=L, ragged=False, text="zipf", V=128256, d=4096, k=16, n_min=3, n_max=8,
             kappa=0, G=1, T=1)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: one chat sequence's decision, latency and launch cost only
        _case("step_1x2k", "step", 1, 2048, text="uniform", k=8),
        # a host-driven engine: inputs from pinned memory, the decisions read back each step
        _case("plan_64x8k", "plan", 64, 8192, text="uniform", k=8),
        # the benchmark's headline: a batch of 32K contexts, four micro-batches in turn
        _case("decode_64x32k", "decode", 64, 32768, G=4, T=4),
        # sampling at T > 0 on ragged rows of odd sizes, one batch, the paper's kappa, the [B, k+1, d] states
        _case("sampled_37x9k", "sampled", 37, 9001, ragged=True, text="uniform", k=12, kappa=5, T=8),
        # the paper's W = 10 candidates of D = 20 tokens
        _case("candidates_64x32k", "candidates", 64, 32768, k=20, kappa=5, G=2, T=4, W=10, D=20),
        # code completion at a large batch with the two-layer probe
        _case("mlp_256x16k", "mlp", 256, 16384, text="code", V=152064, d=5120, k=8, G=2, T=4, H1=256),
        # the two-layer probe at the largest batch, short ragged contexts: the contraction weighs most
        _case("mlp_768x4k", "mlp", 768, 4096, ragged=True, d=4096, k=8, T=4, H1=512),
        # long documents, long drafts, the widest n range
        _case("decode_16x128k", "decode", 16, 131072, V=152064, d=5120, k=32, n_min=2, n_max=12, G=4, T=2),
        # the largest: many long ragged contexts (HBM-bound)
        _case("long_96x200k", "decode", 96, 200000, ragged=True, k=16, T=4),
        # prefill with the incremental index
        _case("index_build_64x32k", "index_build", 64, 32768),
        # decoding with the incremental index on long documents
        _case("index_16x128k", "index", 16, 131072, V=152064, d=5120, k=32, n_min=2, n_max=12, G=4, T=4),
        # labels for a batch of training documents
        _case("labels_64x32k", "labels", 64, 32768, ragged=True, n=5),
    ]


def draw(rng):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["step", "plan", "decode", "sampled", "candidates", "mlp", "long", "index_build", "index", "labels"])
    c = _case("", kind, 1, 1)
    del c["name"]
    n_min = rng.choice([2, 3, 3, 4])
    c.update(ragged=rng.random() < 0.6, text=rng.choice(["zipf", "uniform", "code"]), V=rng.choice([32000, 128256, 152064]),
             d=rng.choice([2048, 4096, 5120, 8192]), k=rng.choice([4, 8, 11, 16, 32]), n_min=n_min,
             n_max=rng.randint(max(5, n_min), 12), kappa=rng.choice([0, 5]))
    rows = {"step": (1, 16), "plan": (8, 128), "decode": (1, 128), "sampled": (1, 128), "candidates": (4, 64),
            "mlp": (16, 768), "long": (1, 96), "index_build": (1, 64), "index": (1, 128), "labels": (1, 64)}[kind]
    toks = {"step": (512, 16384), "plan": (1024, 16384), "decode": (2048, 200000), "sampled": (1024, 65536),
            "candidates": (4096, 65536), "mlp": (1024, 16384), "long": (200000, 1000000), "index_build": (1024, 131072),
            "index": (2048, 131072), "labels": (1024, 262144)}[kind]
    most = {"long": 19_200_000, "mlp": 4_200_000}.get(kind, 2_100_000)  # tokens in all rows
    B = logint(*rows)
    c.update(B=B, L=logint(toks[0], max(toks[0], min(toks[1], most // B))))
    if kind == "long":
        c["B"] = max(1, min(B, most // c["L"]))
        c.update(kind="decode", T=4)
    elif kind in ("decode", "mlp", "index", "candidates"):
        c.update(G=rng.choice([1, 2, 4]), T=4)
    elif kind == "sampled":
        c.update(T=8)
    if kind == "candidates":
        c.update(W=rng.randint(2, 16), D=rng.choice([8, 13, 20, 32]))
        c["k"] = max(c["k"], c["D"])
    if kind == "mlp":
        c["H1"] = rng.choice([64, 100, 256, 384, 512])
    if kind == "labels":
        c["n"] = rng.randint(3, 8)
    return c


# ---------------------------------------------------------------- inputs
def _zipf(V, shape, gen):
    """Zipf(1.1) ids: the rank by inverse CDF, the id by a fixed odd stride over the vocabulary."""
    cdf = torch.cumsum(torch.arange(1, V + 1, device="cuda", dtype=torch.float64).pow_(-1.1), 0)
    cdf = (cdf / cdf[-1]).float()
    r = torch.searchsorted(cdf, torch.rand(shape, device="cuda", generator=gen)).clamp_(max=V - 1)
    return (r * 7919 + 13) % V


def _text(c, R, L, n_future, gen):
    """int64 [R, L + n_future]: R rows of context and the target's stream after it (lengths end at lens)."""
    V, total = c["V"], L + n_future

    def rnd(hi, shape):
        return torch.randint(0, hi, shape, device="cuda", generator=gen)

    if c["text"] == "code":
        blocks = rnd(V, (R, 8, 200))
        order = rnd(8, (R, (total + 199) // 200))
        x = torch.gather(blocks.view(R, 1600), 1,
                         (order[:, :, None] * 200 + torch.arange(200, device="cuda")).reshape(R, -1))[:, :total]
        edit = torch.rand(x.shape, device="cuda", generator=gen) < 0.01
        return torch.where(edit, rnd(V, x.shape), x)
    x = _zipf(V, (R, total), gen) if c["text"] == "zipf" else rnd(V, (R, total))
    # planted copies: 16 spans a row, about a tenth of the context
    pos = torch.arange(total, device="cuda").expand(R, total)
    src = pos.clone()
    span = max(16, min(512, L // 160))
    for _ in range(16):
        dst = rnd(L - span, (R, 1)).clamp_(min=1)
        back = (torch.rand((R, 1), device="cuda", generator=gen) * dst).long() + 1
        hit = (pos >= dst) & (pos < dst + span)
        src = torch.where(hit & (pos - back >= 0), pos - back, src)
    return torch.gather(x, 1, src)


def _inputs(c, seed):
    """Every input of the case, on the GPU, from the seed alone."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) * 1000003 + c["B"] * 8191 + c["L"])
    B, L, G, T, k, d = c["B"], c["L"], c["G"], c["T"], c["k"], c["d"]
    R = G * B
    D = c.get("D", k)
    grow = T * (D + 1) if c["kind"] in GRAPHED or c["kind"] == "plan" else 0
    cap = (L + grow + 3) // 4 * 4
    lens = torch.full((R,), L, device="cuda", dtype=torch.int64)
    if c["ragged"]:
        lens = torch.randint(max(16, L // 2), L + 1, (R,), device="cuda", generator=gen)
    x = _text(c, R, L, grow + D + 2, gen)
    pos = torch.arange(x.shape[1], device="cuda").expand(R, -1)
    if c["text"] != "code":
        # half of the rows end (and go on) inside a copy of an earlier span; one token in ten of the
        # continuation departs from it
        inside = torch.rand((R, 1), device="cuda", generator=gen) < 0.5
        off = (torch.rand((R, 1), device="cuda", generator=gen) * (lens[:, None] * 0.8)).long() + lens[:, None] // 10 + 1
        back = pos - off
        tail = inside & (pos >= lens[:, None] - 40) & (back >= 0)
        edit = (torch.rand(x.shape, device="cuda", generator=gen) < 0.1) & (pos >= lens[:, None])
        x = torch.where(tail & ~edit, torch.gather(x, 1, back.clamp(min=0)), x)
    ctx = torch.where(pos[:, :cap] < lens[:, None], x[:, :cap], torch.zeros_like(x[:, :cap])).to(torch.int32).contiguous()
    s = dict(ctx=ctx, lens=lens.to(torch.int32), cap=cap)
    if c["kind"] == "labels":
        return s
    rows = k + 1 if c["kind"] == "sampled" else 1
    s["hidden"] = torch.randn((T, G, B, rows, d), device="cuda", generator=gen).to(torch.bfloat16)
    if c["kind"] == "mlp":
        H1 = c["H1"]
        w = torch.cat([(torch.randn((H1, d), device="cuda", generator=gen) / math.sqrt(d)).reshape(-1),
                       torch.randn(H1, device="cuda", generator=gen) / math.sqrt(H1)])
    else:
        w = torch.randn(d, device="cuda", generator=gen) / math.sqrt(d)
    s["probe_w"] = w.to(torch.bfloat16)
    if c["kind"] in ("step", "index_build"):
        return s
    # per iteration: the target's tokens, the draft to verify and its length; cur = tokens appended so far
    s["draft"], s["target"], s["dlen"], s["arow"] = [], [], [], []
    s["p"], s["q"], s["u"], s["cand_len"] = [], [], [], []
    cur = torch.zeros(R, device="cuda", dtype=torch.int64)
    W = c.get("W", 1)
    for _ in range(T):
        at = (lens + cur)[:, None] + torch.arange(D + 1, device="cuda")
        g = torch.gather(x, 1, at.clamp(max=x.shape[1] - 1))                       # [R, D + 1]
        agree = torch.rand((R, W, D), device="cuda", generator=gen) < 0.75
        other = torch.randint(0, c["V"], (R, W, D), device="cuda", generator=gen)
        dr = torch.where(agree, g[:, None, :D].expand(-1, W, -1), other)
        dl = torch.where(torch.rand((R, W), device="cuda", generator=gen) < 0.5, min(6, D), D)
        live = torch.arange(D, device="cuda") < dl[:, :, None]
        tgt = g
        if c["kind"] == "sampled":
            same = dr[:, 0] == g[:, :D]
            p = torch.where(same, 0.9, 0.05).float()
            q = torch.where(dl[:, :1] == D, 1.0, 0.8).expand(-1, D).float().contiguous()
            u = torch.rand((R, D), device="cuda", generator=gen)
            ok = (u * q) < p
            s["p"].append(p), s["q"].append(q), s["u"].append(u)
            acc = (ok & live[:, 0]).long().cumprod(1).sum(1)
        elif W > 1:
            nc = torch.where(torch.rand(R, device="cuda", generator=gen) < 0.5, 1, W)
            used = torch.arange(W, device="cuda") < nc[:, None]
            per = ((dr == g[:, None, :D]) & live & used[:, :, None]).long().cumprod(2).sum(2)
            acc = per.max(1).values
            s["cand_len"].append(dl.to(torch.int32).contiguous())
            tgt, dl = g[:, None].expand(-1, W, -1), nc[:, None]
        else:
            acc = ((dr[:, 0] == g[:, :D]) & live[:, 0]).long().cumprod(1).sum(1)
        s["draft"].append(dr.reshape(G, B, W, D).to(torch.int32).contiguous())
        s["target"].append(tgt.reshape(G, B, -1).to(torch.int32).contiguous())
        s["dlen"].append(dl[:, 0].reshape(G, B).to(torch.int32).contiguous())
        s["arow"].append(acc)
        cur = cur + acc + 1
    return s


# ---------------------------------------------------------------- prepare and run
def _params(c, s, stream, ws, index):
    p = bd.switchsd_params()
    p.B, p.cap, p.d, p.k = c["B"], s["cap"], c["d"], c["k"]
    p.n_min, p.n_max, p.kappa, p.logit_tau = c["n_min"], c["n_max"], c["kappa"], 0.0
    mlp = c["kind"] == "mlp"
    p.probe_kind, p.probe_hidden = (bd.PROBE_MLP, c["H1"]) if mlp else (bd.PROBE_LINEAR, 0)
    p.stream = stream.cuda_stream
    # the kernel before each launch is another micro-batch's step, or (one batch) the batch's own last step,
    # which writes the contexts but no hidden state
    if c["kind"] in GRAPHED:
        p.prefetch = bd.PREFETCH_PROBE | (bd.PREFETCH_CONTEXT if c["G"] > 1 else 0)
    if c["kind"] == "sampled":
        p.hidden_rows = c["k"] + 1
    p.index = index.handle if index is not None else None
    p.workspace, p.workspace_bytes = ws.data_ptr(), ws.numel()
    return p


def _ok(code):
    if code != bd.OK:
        raise RuntimeError(f"a controller call failed: {code} ({bd.strerror(code)})")


def _prepare_graph(c, s):
    lib = bd.load()
    B, G, T, k, cap = c["B"], c["G"], c["T"], c["k"], s["cap"]
    W, D = c.get("W", 1), c.get("D", k)
    cand = c["kind"] == "candidates"
    stream = torch.cuda.Stream()
    lens = s["lens"].clone()

    def ints(*shape):
        return torch.zeros(shape, dtype=torch.int32, device="cuda")

    o = dict(mode=ints(T, G, B), score=torch.zeros((T, G, B), dtype=torch.float32, device="cuda"), match_n=ints(T, G, B),
             match_end=ints(T, G, B), accept=ints(T, G, B), status=ints(T, G, B))
    if cand:
        o.update(cand=ints(T, G, B, W, D), cand_len=ints(T, G, B, W), ncand=ints(T, G, B), choice=ints(T, G, B))
    else:
        o.update(draft=ints(T, G, B, k), len=ints(T, G, B))
    keep, calls = [], []
    torch.cuda.synchronize()
    for g in range(G):
        need = bd.switchsd_workspace_bytes(B, bd.PROBE_MLP, c["H1"], c["d"]) if c["kind"] == "mlp" else 0
        ws = torch.empty(max(need, 16), dtype=torch.uint8, device="cuda")  # one workspace a micro-batch
        index = None
        if c["kind"] == "index":
            index = bd.NgramIndex(B, cap, c["n_min"], c["n_max"])
            index.build(s["ctx"][g * B:(g + 1) * B], s["lens"][g * B:(g + 1) * B], stream=stream)
        for t in range(T):
            p = _params(c, s, stream, ws, index)
            p.out_match_n, p.out_match_end = o["match_n"][t, g].data_ptr(), o["match_end"][t, g].data_ptr()
            p.status = o["status"][t, g].data_ptr()
            keep.append((p, ws, index))
            dr, tg, dl, ac = s["draft"][t][g], s["target"][t][g], s["dlen"][t][g], o["accept"][t, g]
            state = (s["ctx"][g * B:].data_ptr(), lens[g * B:].data_ptr(), s["hidden"][t, g].data_ptr(),
                     s["probe_w"].data_ptr(), ctypes.byref(p))
            outs = (o["mode"][t, g].data_ptr(), o["score"][t, g].data_ptr())
            if cand:
                a = (dr.data_ptr(), tg.data_ptr(), s["cand_len"][t][g * B:].data_ptr(), dl.data_ptr(), ac.data_ptr(),
                     o["choice"][t, g].data_ptr(), *state, W, D, o["cand"][t, g].data_ptr(),
                     o["cand_len"][t, g].data_ptr(), o["ncand"][t, g].data_ptr(), *outs)
                fn = lib.switchsd_verify_candidates_step
            else:
                more = (o["draft"][t, g].data_ptr(), o["len"][t, g].data_ptr(), *outs)
                a = (dr.data_ptr(), tg.data_ptr(), dl.data_ptr(), ac.data_ptr(), *state, *more)
                fn = lib.switchsd_verify_step
                if c["kind"] == "sampled":
                    a = (dr.data_ptr(), s["p"][t].data_ptr(), s["q"][t].data_ptr(), s["u"][t].data_ptr(), *a[1:])
                    fn = lib.switchsd_verify_sampled_step
            calls.append((t, g, fn, a))
    calls.sort(key=lambda e: e[:2])

    def one_pass():
        lens.copy_(s["lens"])  # the batch's start; the contexts' appended tokens are written again
        for _, _, fn, a in calls:
            _ok(fn(*a))

    with torch.cuda.stream(stream):
        one_pass()  # first calls outside the capture
    stream.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        one_pass()
    o.update(ctx=s["ctx"], lens=lens)
    return dict(kind="graph", graph=graph, out=o, keep=(s, keep, calls, stream))


def prepare(case, seed):
    c = case
    s = _inputs(c, seed)
    if c["kind"] in GRAPHED:
        return _prepare_graph(c, s)
    B, k = c["B"], c["k"]
    if c["kind"] == "labels":
        need = int(bd.load().switchsd_labels_workspace_bytes(B, s["cap"]))
        return dict(kind="labels", n=c["n"], s=s, labels=torch.zeros((B, s["cap"]), dtype=torch.uint8, device="cuda"),
                    ws=torch.empty(need, dtype=torch.uint8, device="cuda"))
    sess = Session(s["ctx"].cpu().numpy(), s["lens"].cpu().numpy(),
                   s["probe_w"].view(torch.int16).cpu().numpy().view("uint16"), k=k, n_min=c["n_min"], n_max=c["n_max"],
                   kappa=c["kappa"], d=c["d"], use_index=c["kind"] == "index_build")
    st = dict(kind=c["kind"], sess=sess, hidden=s["hidden"].reshape(B, c["d"]), lens=s["lens"])
    if c["kind"] == "plan":
        sess.vdraft.copy_(s["draft"][0].view(B, k))
        sess.target.copy_(s["target"][0].view(B, k + 1))
        sess.vlen.copy_(s["dlen"][0].view(B))
        st["host"] = st["hidden"].cpu().pin_memory()
        st["dev"] = torch.empty_like(st["hidden"])
        st["results"] = torch.zeros(B * (k + 3), dtype=torch.int32, pin_memory=True)
        st["plan"] = sess.host_plan(st["host"], st["dev"], st["results"], verify=True, debug=True)
    torch.cuda.synchronize()
    return st


def run(state):
    kind = state["kind"]
    if kind == "graph":
        state["graph"].replay()
        return state["out"]
    if kind == "labels":
        s = state["s"]
        bd.switchsd_copy_labels(s["ctx"], s["lens"], state["labels"], n=state["n"], workspace=state["ws"])
        return state["labels"]
    sess = state["sess"]
    if kind == "plan":
        sess.lens.copy_(state["lens"])  # the batch's start
        state["plan"].run(state["host"], state["results"])
        r = state["plan"].results()
        return dict(mode=r["mode"], len=r["len"], accept=r["accept"], draft=r["draft"], score=sess.score,
                    match_n=sess.match_n, match_end=sess.match_end, ctx=sess.ctx, lens=sess.lens)
    if kind == "index_build":
        sess.index.build(sess.ctx, sess.lens)
    sess.step(state["hidden"])
    return dict(mode=sess.mode, len=sess.len, draft=sess.draft, score=sess.score, match_n=sess.match_n,
                match_end=sess.match_end, status=sess.status)


# ---------------------------------------------------------------- work, tolerance, exact
def work(case):
    c = case
    B, L, d, k, n = c["B"], c["L"], c["d"], c["k"], c["G"] * c["T"]
    tokens = B * L * (0.75 if c["ragged"] else 1.0)
    if c["kind"] == "labels":
        return {"bytes": tokens * 4 + B * L, "flops": 0}
    grams = c["n_max"] - c["n_min"] + 1
    small = B * (4 * k + 24)                                   # the step's outputs
    if c["kind"] != "step" and c["kind"] != "index_build":
        small += B * (8 * c.get("W", 1) * c.get("D", k) + 8)   # the verification's inputs
    state, flops = 2 * B * d + 2 * d, 2 * B * d
    if c["kind"] == "sampled":
        small += 12 * B * k
    if c["kind"] == "candidates":
        small += 4 * B * c["W"] * c["D"]
    if c["kind"] == "mlp":
        state, flops = 2 * B * d + 2 * d * c["H1"], 2 * B * d * c["H1"]
    if c["kind"] == "index_build":  # tokens read, one link a position and length written
        return {"bytes": tokens * 4 * (1 + grams) + state + small, "flops": flops}
    # the index reads a row's tail and, per length, a head, a link and the tokens compared
    search = B * (4 * 32 + grams * (8 + 4 * c["n_max"])) if c["kind"] == "index" else tokens * 4
    return {"bytes": n * (search + state + small), "flops": n * flops}


def tolerance(case):
    # every output but the probe's logit is whole and exact; the logit is a sum of d products in 32 bits (seen
    # against 64 bits: 1e-7 for the linear probe, 3e-7 for the two-layer one; a reordered sum differs as much)
    if case["kind"] == "labels":
        return "exact"
    return {"rel": 2e-6, "max": 2e-5} if case["kind"] == "mlp" else {"rel": 1e-6, "max": 1e-5}


def exact(case, seed):
    """The probe's logits in 64 bits; the other outputs are whole numbers."""
    c = case
    if c["kind"] == "labels":
        return None
    s = _inputs(c, seed)
    T, G, B, d = c["T"], c["G"], c["B"], c["d"]
    h, w = s["hidden"], s["probe_w"].double()
    if c["kind"] == "sampled":  # the probed state is row a_b of each row's k + 1
        at = torch.stack(s["arow"]).view(T, G, B, 1, 1).expand(-1, -1, -1, 1, d)
        h = torch.gather(h, 3, at)
    z = []
    for t in range(T):
        ht = h[t].reshape(G * B, d).double()
        if c["kind"] == "mlp":
            H1 = c["H1"]
            z.append(torch.relu(ht @ w[:H1 * d].view(H1, d).T) @ w[H1 * d:])
        else:
            z.append(ht @ w)
    z = torch.stack(z).view(T, G, B)
    return {"score": z if c["kind"] in GRAPHED else z.view(B)}
