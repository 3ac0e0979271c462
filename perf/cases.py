"""The calls whose speed matters to a user of this library, as cases that can be timed.

Three kinds of case:

``step``  what one process of a data-parallel job does with its sparse gradients in an iteration:
          ``own`` workers compress here (0, 1, or several in one call), then ``lists`` sparse sets --
          the own ones and, where there are more, those that came in from other ranks -- are summed
          into a dense buffer (``apply`` = "dense": cleared first, "add": on top of its content) or
          go straight into momentum SGD ("momentum").  ``lists`` = 0: compress only.
``hook``  one layer's gradient compressed by the call that needs no plan and allocates nothing, as a
          gradient hook inside a training framework uses it.
``rows``  the embedding-table server: optimizer step with parity update on the rows of a batch,
          then rows of a failed server rebuilt from the survivors and the parity.

Every result is defined bit for bit (exact selection, fixed order of the sums, one rounding per
operation), so the tolerance is "exact" throughout.
"""
import math

import torch

from paper_2104_01981_b200 import api, ecrm, synth

BERT = sum(synth.numel(s) for s in synth.bert_base_shapes())        # 109,482,240
GPT2 = sum(synth.numel(s) for s in synth.gpt2_medium_shapes())      # 354,823,168


def _step(layout, n, density, own=1, lists=0, apply="dense", dtype="fp32", threshold=False, private=False):
    return {"kind": "step", "layout": layout, "n": n, "density": density, "own": own, "lists": lists,
            "apply": apply, "dtype": dtype, "threshold": threshold, "private": private}


def listed():
    return [
        # a small model, or one bucket of a larger one, on one worker: latency of compress and decode
        dict(_step("normal", 1 << 20, 0.01, lists=1), name="step_1m"),
        # one layer of odd size inside a gradient hook that may not allocate
        {"name": "hook_2m4", "kind": "hook", "n": 2_361_599, "density": 0.01},
        # layer-wise sparsification of a convolutional network: 161 tensors, most of them tiny
        dict(_step("resnet50", 0, 0.001), name="topk_resnet50"),
        # global top-k of a transformer, heavy-tailed gradient: the headline workload
        dict(_step("student", BERT, 0.01, private=True), name="topk_bert"),
        # the same with mixed-precision training's bfloat16 gradient
        dict(_step("student", BERT, 0.01, dtype="bf16", private=True), name="topk_bert_bf16"),
        # the transformer layer by layer, at a density of the first epochs, before it is lowered
        dict(_step("bert", 0, 0.05), name="topk_bert_layers_5pct"),
        # sampled threshold instead of exact top-k, one tensor
        dict(_step("student", BERT, 0.01, threshold=True), name="threshold_bert"),
        # eight workers on one GPU, layer-wise, optimizer fused behind the sum
        dict(_step("resnet50", 0, 0.001, own=8, lists=8, apply="momentum", private=True), name="step_resnet50_8w"),
        # the same workers in threshold mode: lists of varying length, dense sum
        dict(_step("resnet50", 0, 0.001, own=8, lists=8, threshold=True), name="step_resnet50_8w_thr"),
        # one of sixteen ranks: own compress, then the sixteen gathered lists summed
        dict(_step("outliers", GPT2, 0.001, lists=16, private=True), name="step_gpt2_16w"),
        # thirty-two gathered lists summed
        dict(_step("student", BERT, 0.01, own=0, lists=32), name="decode_bert_32w"),
        # embedding server during a recovery: a batch's update with parity, and reads of lost rows
        {"name": "rows_2m", "kind": "rows", "table": 2_000_000, "batch": 200_003, "reads": 50_001, "dim": 128, "k": 4,
         "optimizer": "adagrad"},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """Flat gradients of 100 thousand to 355 million elements, layered ones of 161 to 200 tensors or
    a ragged dozen, densities of 0.1 to 5 %, one to 32 workers; layers of 20 thousand to 16 million
    elements; batches of a thousand to 400 thousand rows."""
    most = max(work(c)["bytes"] for c in listed())
    while True:
        kind = rng.choice(["step"] * 8 + ["hook", "rows"])
        if kind == "hook":
            c = {"kind": "hook", "n": int(_log(rng, 2e4, 1 << 24)), "density": _log(rng, 1e-3, 5e-2)}
        elif kind == "rows":
            table = int(_log(rng, 5e4, 2e6))
            c = {"kind": "rows", "table": table, "batch": int(min(_log(rng, 1e3, 4e5), table // 2)),
                 "reads": int(min(_log(rng, 1e3, 2e5), table // 2)), "dim": rng.choice([32, 64, 128]),
                 "k": rng.choice([2, 3, 4, 8]), "optimizer": rng.choice(["adagrad", "momentum"])}
        else:
            layout = rng.choice(["normal", "student", "outliers", "resnet50", "bert", "ragged"])
            n = 0 if layout in ("resnet50", "bert") else int(_log(rng, 1e5, GPT2))
            own = rng.choice([1, 1, 1, 0, rng.randint(2, 8)])
            threshold = own > 0 and rng.random() < 0.25
            lists = own if threshold else rng.choice([own, int(round(_log(rng, max(own, 1), 32)))])
            if own == 1 and rng.random() < 0.5:
                lists = 0
            if own + lists == 0:
                continue
            density = _log(rng, 1e-3, 5e-2)
            # bfloat16 gradients: one worker, top-k, plans that the fused kernels take
            bf16 = own == 1 and not threshold and (layout == "resnet50" or layout in ("normal", "student", "outliers")
                                                   and n * density < 2.5e6)
            c = _step(layout, n, density, own, lists, rng.choice(["dense", "dense", "add", "momentum"]),
                      "bf16" if bf16 and rng.random() < 0.4 else "fp32", threshold, rng.random() < 0.5)
        if work(c)["bytes"] <= most:
            return c


# --------------------------------------------------------------------------- inputs
def _sizes(case):
    layout, n = case["layout"], case["n"]
    if layout == "resnet50":
        return [synth.numel(s) for s in synth.resnet50_shapes()]
    if layout == "bert":
        return [synth.numel(s) for s in synth.bert_base_shapes()]
    if layout == "ragged":                          # a dozen tensors, the largest about 40 times the smallest
        weight = [(1 + i * 7919 % 13) ** 1.5 for i in range(12)]
        sizes = [max(1, int(n * x / sum(weight))) for x in weight]
        sizes[0] += n - sum(sizes)
        return sizes
    return [n]


def _workload(case):
    """The case's gradient as a workload of paper_2104_01981_b200.synth, and its standard deviation
    per tensor."""
    sizes = _sizes(case)
    if case["layout"] == "student":
        return synth.Workload("case", 12, sizes, case["density"], 1, 1, "student_t3", sigma=0.02), [0.02 * 3 ** 0.5]
    if case["layout"] == "outliers":
        return synth.Workload("case", 14, sizes, case["density"], 1, 1, "normal_outliers", sigma=0.02), [0.02 * 1.12]
    if case["layout"] == "normal":
        return synth.Workload("case", 10, sizes, case["density"], 1, 1, "normal", sigma=1.0), [1.0]
    if case["layout"] == "ragged":
        scales = [1.0 / math.sqrt(1 + s % 977) for s in sizes]
    else:
        shapes = synth.resnet50_shapes() if case["layout"] == "resnet50" else synth.bert_base_shapes()
        scales = [1.0 / math.sqrt(synth.fan_in(s)) for s in shapes]
    return synth.Workload("case", 11, sizes, case["density"], 1, 1, "layer_normal", scales=scales), scales


def _residual(sizes, stds, density, gen):
    """Residual in the middle of a run.  Under error feedback an entry's residual is a random walk
    that starts again from 0 when it reaches the threshold T; it gets there after 1/density steps on
    average, so T = std / sqrt(density), and the walk's stationary law is triangular on (-T, T)."""
    n = sum(sizes)
    r = torch.empty(n, device="cuda").uniform_(generator=gen)
    chunk = 1 << 25
    for lo in range(0, n, chunk):
        v = r[lo:lo + chunk]
        v.sub_(torch.empty_like(v).uniform_(generator=gen))
    off = 0
    for s, std in zip(sizes, stds):
        r[off:off + s].mul_(std / math.sqrt(density))
        off += s
    return r


def _foreign_lists(sizes, ks, count, gen):
    """Sparse sets of other workers: per tensor the k largest of a score that is 20 % correlated
    between workers, as gradients of one model on different batches are."""
    n = sum(sizes)
    common = torch.empty(n, device="cuda").normal_(generator=gen).mul_(0.5)
    score = torch.empty(n, device="cuda")
    lists = []
    for _ in range(count):
        score.normal_(generator=gen).add_(common)
        parts, off = [], 0
        for s, k in zip(sizes, ks):
            parts.append(score[off:off + s].abs().topk(k, sorted=False).indices.sort().values + off)
            off += s
        idx = torch.cat(parts)
        lists.append((idx.to(torch.int32), score[idx].mul(0.1)))
    return lists


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed * 7919 + 17)
    if case["kind"] == "hook":
        n = case["n"]
        w, stds = _workload({"layout": "normal", "n": n, "density": case["density"]})
        k = max(1, math.ceil(n * case["density"]))
        return {"case": case, "grad": synth.gradient(w, 0, 0, device="cuda", seed0=seed),
                "resid": _residual([n], stds, case["density"], gen), "k": k,
                "idx": torch.zeros(k, dtype=torch.int32, device="cuda"), "val": torch.zeros(k, device="cuda"),
                "status": torch.zeros(1, dtype=torch.int32, device="cuda")}
    if case["kind"] == "rows":
        return _prepare_rows(case, gen)

    w, stds = _workload(case)
    sizes, own, count = w.sizes, case["own"], case["lists"]
    plan = api.Plan(sizes, case["density"], mode=api.GC_THRESHOLD if case["threshold"] else api.GC_TOPK, device=0)
    if case["private"]:
        plan.set_option(api.GC_OPT_WORKSPACE_PRIVATE, 1)
    st = {"case": case, "plan": plan, "ws": [plan.alloc_workspace() for _ in range(max(own, 1))]}
    st["grad"] = [synth.gradient(w, i, 0, device="cuda", seed0=seed) for i in range(own)]
    if case["dtype"] == "bf16":
        st["grad"] = [g.to(torch.bfloat16) for g in st["grad"]]
    st["resid"] = [_residual(sizes, stds, case["density"], gen) for _ in range(own)]
    outs = [(torch.zeros(plan.total_cap, dtype=torch.int32, device="cuda"), torch.zeros(plan.total_cap, device="cuda"),
             torch.zeros(2 * plan.n_tensors, dtype=torch.int32, device="cuda")) for _ in range(own)]
    st["idx"], st["val"], st["cnt"] = ([o[i] for o in outs] for i in range(3))
    if count:
        more = _foreign_lists(sizes, plan.tensor_k(), count - own, gen) if count > own else []
        st["all_idx"] = st["idx"] + [m[0] for m in more]
        st["all_val"] = st["val"] + [m[1] for m in more]
        if case["apply"] == "momentum":
            st["param"] = torch.empty(plan.total_n, device="cuda").normal_(generator=gen).mul_(0.05)
            st["velocity"] = torch.empty(plan.total_n, device="cuda").normal_(generator=gen).mul_(0.01)
        else:
            st["dense"] = torch.zeros(plan.total_n, device="cuda")
    return st


def _prepare_rows(case, gen):
    table, dim, k = case["table"], case["dim"], case["k"]

    def some_rows(m):                               # distinct rows in no order, as a batch's unique leaves them
        return torch.randperm(table, generator=gen, device="cuda")[:m].to(torch.int32)

    def shard(scale):
        return torch.empty(table, dim, device="cuda").normal_(generator=gen).mul_(scale)

    shards = [shard(0.01) for _ in range(k)]        # shards[0] is updated; shard 0 of the reads is the lost one
    p_entry = torch.zeros(table, dim, device="cuda")
    for s in shards:
        p_entry.add_(s)
    state = shard(0.1).square_()
    return {"case": case, "entry": shards[0], "others": shards[1:], "state": state, "p_entry": p_entry,
            "p_state": state * k, "rows": some_rows(case["batch"]), "prow": some_rows(case["batch"]),
            "grad": torch.empty(case["batch"], dim, device="cuda").normal_(generator=gen).mul_(0.05),
            "reads": some_rows(case["reads"]), "out": torch.zeros(case["reads"], dim, device="cuda"),
            "bad": torch.zeros(1, dtype=torch.int32, device="cuda")}


# --------------------------------------------------------------------------- one pass
def run(st):
    case = st["case"]
    if case["kind"] == "hook":
        api.compress_noalloc(st["grad"], st["resid"], case["n"], st["k"], st["idx"], st["val"], st["status"])
        return [st["idx"], st["val"], st["resid"], st["status"]]
    if case["kind"] == "rows":
        opt, hyper = (ecrm.ECRM_ADAGRAD, 1e-8) if case["optimizer"] == "adagrad" else (ecrm.ECRM_MOMENTUM, 0.9)
        ecrm.rows_step_parity(opt, st["rows"], st["prow"], st["grad"], st["entry"], st["state"], st["p_entry"],
                              st["p_state"], 0.01, hyper, st["bad"])
        ecrm.degraded_read(st["reads"], None, st["others"], st["p_entry"], st["out"], st["bad"])
        return [st["entry"], st["state"], st["p_entry"], st["p_state"], st["out"], st["bad"]]

    plan, own, count = st["plan"], case["own"], case["lists"]
    out = []
    if own == 1:
        call = plan.compress_bf16 if case["dtype"] == "bf16" else plan.compress
        call(st["grad"][0], st["resid"][0], st["idx"][0], st["val"][0], st["cnt"][0], st["ws"][0])
    elif own > 1:
        plan.compress_workers(st["grad"], st["resid"], st["idx"], st["val"], st["cnt"], st["ws"])
    if own:
        out += st["idx"] + st["val"] + st["cnt"] + st["resid"]
    if count:
        cnt = st["cnt"] if case["threshold"] else None
        if case["apply"] == "momentum":
            plan.decompress_apply_momentum(st["all_idx"], st["all_val"], cnt, st["param"], st["velocity"], 0.05, 0.9,
                                           1.0 / count, st["ws"][0])
            out += [st["param"], st["velocity"]]
        else:
            plan.decompress_accumulate(st["all_idx"], st["all_val"], cnt, st["dense"], case["apply"] == "dense",
                                       st["ws"][0])
            out.append(st["dense"])
    return out


def work(case):
    if case["kind"] == "hook":
        n, k = case["n"], math.ceil(case["n"] * case["density"])
        return {"bytes": 12 * n + 8 * k, "flops": n}
    if case["kind"] == "rows":
        m, q, dim, k = case["batch"], case["reads"], case["dim"], case["k"]
        # the batch: gradient, entry, state and both parities read, the last four written
        return {"bytes": m * (9 * 4 * dim + 8) + q * ((k + 1) * 4 * dim + 4), "flops": 7 * m * dim + (k - 1) * q * dim}
    sizes = _sizes(case)
    n, k = sum(sizes), sum(min(s, max(1, math.ceil(s * case["density"]))) for s in sizes)
    own, count = case["own"], case["lists"]
    fold = own * ((10 if case["dtype"] == "bf16" else 12) * n + 8 * k)
    aggregate = {"dense": 4, "add": 8, "momentum": 16}[case["apply"]] * n + 8 * count * k if count else 0
    return {"bytes": fold + aggregate,
            "flops": own * n + count * k + (4 * n if count and case["apply"] == "momentum" else 0)}


def tolerance(case):
    return "exact"
