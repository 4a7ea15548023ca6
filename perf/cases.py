"""The work that users of this library have it do, as measurable cases.

A case is one call, or one run of calls, through the public binding
(``paper_2105_01196_gb300.ebic``), at the sizes of the repository's workloads (tiny 200 x 20,
default 10,000 x 100, batched 20,000 x 500, tie-heavy 60,000 x 1,000, the serving stream's
1,000-50,000 x 20-500) and at ragged sizes between them:

  sweep    one population evaluated on a loaded matrix: a program with its own search calls this
           once per iteration, with host arrays or device tensors;
  noalloc  the same evaluation from caller memory only, as a serving process calls it;
  pairs    a matrix loaded, its pair bitmap built, the pair counts read: what every new matrix
           costs before the first bitmap evaluation;
  job      a whole search: matrix loaded, initial population, the generations, the top list and
           the row masks of its biclusters;
  served   the same through the job server, from a host matrix, one job waited for.

Values: a normal background (hardly any ties), or log-normal rounded to 0.1 (ties in every column
pair), both with planted trend biclusters.
"""

import math

import numpy as np
import torch

from paper_2105_01196_gb300 import ebic


def _case(name, kind, rows, cols, pop, lo, hi, num, den, neg, **more):
    c = dict(name=name, kind=kind, rows=rows, cols=cols, pop=pop, lo=lo, hi=hi, num=num, den=den,
             neg=neg, gens=0, data="normal", ties=0, kept=0, host=0, colmajor=0, ahead="none")
    c.update(more)
    return c


def listed():
    return [
        # The smallest call: a toy matrix and population from host arrays, exact upward trends.
        # Launches, copies and round trips are all of it.
        _case("sweep-tiny-host", "sweep", 200, 20, 64, 2, 6, 1, 1, 0, host=1),
        # One iteration of an own search at the default scale, device tensors, the form AUTO
        # takes on a matrix that is evaluated only a few times (8-bit rank codes).
        _case("sweep-default", "sweep", 10_000, 100, 800, 2, 20, 85, 100, 1),
        # The same at the batched scale with a ragged row count, for a program that tunes once
        # and then evaluates many populations.
        _case("sweep-batched-tuned", "sweep", 20_001, 500, 4_096, 2, 64, 85, 100, 1, ahead="tune"),
        # The largest sweep: the tie-heavy workload on its pair bitmap (7.5 GB).
        _case("sweep-tieheavy-bitmap", "sweep", 60_000, 1_000, 8_192, 2, 64, 85, 100, 1,
              data="rounded", ahead="bitmap"),
        # The trend variants (ties hold, comparison with the last kept value), which have the
        # direct form only (16-bit rank codes).
        _case("sweep-lastkept", "sweep", 9_999, 333, 1_000, 2, 30, 9, 10, 1, data="rounded",
              ties=1, kept=1),
        # More columns than rank codes cover: the direct form over the order keys.
        _case("sweep-wide", "sweep", 5_001, 1_500, 512, 2, 40, 85, 100, 1),
        # Evaluation without allocation, at the default scale.
        _case("noalloc-default", "noalloc", 10_000, 100, 800, 2, 20, 85, 100, 1),
        # Preparing a new column-major matrix with ragged sizes for the bitmap form.
        _case("pairs-ragged", "pairs", 33_333, 777, 0, 0, 0, 1, 1, 1, colmajor=1),
        # The default search: 100 generations of 800 individuals.
        _case("job-default", "job", 10_000, 100, 800, 2, 20, 85, 100, 1, gens=100),
        # The batched search: 200 generations of 4,096 individuals.
        _case("job-batched", "job", 20_000, 500, 4_096, 2, 64, 85, 100, 1, gens=200),
        # The benchmark's headline step: the tie-heavy search, tuned beforehand.
        _case("job-tieheavy-tuned", "job", 60_000, 1_000, 8_192, 2, 64, 85, 100, 1, gens=100,
              data="rounded", ahead="tune"),
        # One job of the serving stream, from a host matrix of odd size through the server.
        _case("served-job", "served", 13_579, 247, 800, 2, 20, 85, 100, 1, gens=50, host=1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["sweep", "sweep", "sweep", "noalloc", "pairs", "job", "job", "served"])
    served = kind == "served"
    rows = _log(rng, 1_000, 50_000) if served else _log(rng, 200, 60_000)
    cols = _log(rng, 20, 500) if served else _log(rng, 20, 1_000)
    pop = 800 if served else _log(rng, 64, 8_192)
    if kind == "sweep" and rng.random() < 0.15:  # beyond the rank codes
        rows, cols, pop = _log(rng, 200, 5_000), rng.randint(1_025, 1_500), _log(rng, 64, 1_024)
    hi = min(rng.choice([6, 20, 40, 64]), cols)
    num, den = rng.choice([(85, 100), (85, 100), (9, 10), (3, 4), (1, 1)])
    more = dict(data=rng.choice(["normal", "rounded"]))
    if kind in ("job", "served"):
        more["gens"] = 50 if served else rng.randint(20, 100)
    if kind == "sweep":
        more["host"] = int(rng.random() < 0.3)
        more["ahead"] = rng.choice(["none", "bitmap", "tune"]) if cols <= 1_024 else "none"
        more["ties"] = int(rng.random() < 0.2)
        if more["ahead"] == "none":
            more["kept"] = int(rng.random() < 0.2)
    if kind in ("pairs", "job"):
        more["colmajor"] = int(rng.random() < 0.3)
    if kind == "job":
        more["ahead"] = rng.choice(["none", "none", "tune"])
    if served:
        more["host"] = 1
    if kind == "pairs":
        pop, hi, num, den = 0, 0, 1, 1
    c = _case("", kind, rows, cols, pop, 2 if hi else 0, hi, num, den, int(rng.random() < 0.75),
              **more)
    del c["name"]
    return c


# ------------------------------------------------------------------------------------- inputs

def _matrix(case, g):
    """float32 [rows, cols] on the GPU: the background with planted biclusters of 1-8% of the rows
    (their values rise by 0.5-1.5 per column of the planted order, half of them reversed)."""
    R, C, dev = case["rows"], case["cols"], "cuda"
    rounded = case["data"] == "rounded"
    x = torch.randn(R, C, generator=g, device=dev)
    if rounded:
        x = x.exp_()
    for b in range(max(2, min(20, C // 20))):
        share = torch.rand(2, generator=g, device=dev).tolist()
        nr = max(2, int(R * (0.01 + 0.07 * share[0])))
        nc = max(2, min(C, int(4 + share[1] * min(40, C // 4))))
        rows = torch.randperm(R, generator=g, device=dev)[:nr]
        order = torch.randperm(C, generator=g, device=dev)[:nc]
        steps = 0.5 + torch.rand(nr, nc, generator=g, device=dev)
        start = torch.randn(nr, 1, generator=g, device=dev)
        vals = start + steps.cumsum(1) + 0.1 * torch.randn(nr, nc, generator=g, device=dev)
        if rounded:  # onto the positive scale
            vals = vals - vals.amin(1, keepdim=True) + start.exp()
        x[rows[:, None], order.flip(0) if b % 2 else order] = vals
    if rounded:
        x = (x * 10).round_() / 10
    return x.contiguous()


def _population(case, g):
    """CSR population: lengths uniform in [lo, hi], distinct columns drawn uniformly."""
    P, C, hi = case["pop"], case["cols"], case["hi"]
    lens = torch.randint(case["lo"], hi + 1, (P,), generator=g, device="cuda")
    cols = torch.rand(P, C, generator=g, device="cuda").topk(hi, dim=1).indices
    keep = torch.arange(hi, device="cuda")[None, :] < lens[:, None]
    off = torch.zeros(P + 1, dtype=torch.int32, device="cuda")
    off[1:] = lens.cumsum(0)
    return cols[keep].to(torch.int32).contiguous(), off


def _params(case, seed):
    f = dict(neg_trends=case["neg"], ratio_num=case["num"], ratio_den=case["den"],
             non_strict=case["ties"], last_kept=case["kept"], seed=seed & 0x7FFFFFFF)
    if case["gens"]:
        top = max(10, min(20, case["cols"] // 20))
        f.update(pop_size=case["pop"], max_len=case["hi"], init_min_len=case["lo"],
                 init_max_len=case["hi"], n_biclusters=top, elite=top, tabu_hit_limit=0)
    return ebic.Params.make(**f)


class _State:
    """What a user's program holds between calls."""

    def __del__(self):
        for handle in (getattr(self, "ctx", None), getattr(self, "server", None)):
            if handle is not None:
                handle.close()


def prepare(case, seed):
    s = _State()
    s.case = case
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    x = _matrix(case, g)
    s.params = _params(case, seed)
    if case["pop"]:
        s.col_idx, s.offsets = _population(case, g)
    kind = case["kind"]
    if kind in ("sweep", "noalloc") and not case["host"]:
        s.outs = [torch.zeros(case["pop"], dtype=torch.int32, device="cuda") for _ in range(3)]
        s.outs.append(torch.zeros(case["pop"], dtype=torch.int64, device="cuda"))
    if kind == "noalloc":
        s.x = x.t().contiguous()
    elif kind == "served":
        s.x = x.cpu().numpy()
        s.server = ebic.Server(0, hbm_budget_bytes=16 << 30, max_running=8)
    else:
        s.layout = ebic.COL_MAJOR if case["colmajor"] else ebic.ROW_MAJOR
        s.x = x.t().contiguous() if case["colmajor"] else x
        torch.cuda.synchronize()
        s.ctx = ebic.Context(0)
        if kind == "pairs":
            s.counts = torch.zeros(case["cols"], case["cols"], dtype=torch.int64, device="cuda")
        if kind == "sweep" or case["ahead"] != "none":
            s.ctx.load_matrix(s.x, s.layout)
        if case["ahead"] == "bitmap":
            s.ctx.build_bitmap()
        if case["ahead"] == "tune":  # for the sweeps that the program goes on to make
            s.ctx.autotune(s.col_idx, s.offsets, s.params, (case["gens"] or 100) + 2)
    if kind == "sweep" and case["host"]:
        s.col_idx, s.offsets = s.col_idx.cpu().numpy(), s.offsets.cpu().numpy()
    torch.cuda.synchronize()
    return s


# ------------------------------------------------------------------------------------- the pass

def _top(entries):
    """A top list as arrays: columns (padded with -1), lengths, fitness, keys, row counts."""
    cols = np.full((len(entries), ebic.MAX_LEN), -1, np.int32)
    for k, e in enumerate(entries):
        cols[k, :len(e["cols"])] = e["cols"]
    return {"cols": cols, "len": np.array([len(e["cols"]) for e in entries], np.int32),
            "fitness": np.array([e["f"] for e in entries], np.uint64).view(np.int64),
            "key": np.array([e["h"] for e in entries], np.uint64).view(np.int64),
            "rows": np.array([(e["rows_pos"], e["rows_neg"], e["rows_any"]) for e in entries],
                             np.int32)}


def run(s):
    kind = s.case["kind"]
    if kind == "sweep":
        if s.case["host"]:
            pos, neg, either, fit = s.ctx.eval_population(s.col_idx, s.offsets, s.params)
            return pos, neg, either, fit.view(np.int64)
        return s.ctx.eval_population(s.col_idx, s.offsets, s.params, *s.outs)
    if kind == "noalloc":
        return ebic.ebic_eval_population_noalloc(s.x, s.col_idx, s.offsets, s.params, *s.outs)
    if kind == "pairs":
        s.ctx.load_matrix(s.x, s.layout)
        s.ctx.build_bitmap()
        return s.ctx.copy_pair_counts(s.counts)
    if kind == "served":
        r = s.server.wait(s.server.submit(s.x, s.params, s.case["gens"]))
        if r["status"]:
            raise RuntimeError(f"the job ended with status {r['status']}")
        return {"generations": r["gens_done"], "evaluated": r["n_evaluated"], **_top(r["top"])}
    s.ctx.load_matrix(s.x, s.layout)
    r = s.ctx.run_generations(s.params, s.case["gens"])
    out = {"generations": r.gens_done, "evaluated": r.n_evaluated, "hits": r.last_hits}
    out.update(_top(s.ctx.toplist()))
    out["masks"] = s.ctx.extract_biclusters(s.case["rows"])
    return out


# ------------------------------------------------------------------------------------- its size

def work(case):
    """The matrix and the population read once, the results written once; one comparison per row,
    consecutive pair and direction (of a search, whose lengths evolve: one pair per individual)."""
    R, C, P, G = case["rows"], case["cols"], case["pop"], case["gens"]
    both = 1 + case["neg"]
    pairs = (case["lo"] + case["hi"]) / 2 - 1
    if case["kind"] == "pairs":
        return {"bytes": 4.0 * R * C + C * C * math.ceil(R / 128) * 16, "flops": float(R) * C * C}
    if G:
        masks = (math.ceil(R / 128) * 16 + 300) * max(10, min(20, C // 20))
        return {"bytes": 4.0 * R * C + masks, "flops": float(R) * P * both * (pairs + G)}
    return {"bytes": 4.0 * R * min(C, P * (pairs + 1)) + P * (4 * (pairs + 1) + 24),
            "flops": float(R) * P * pairs * both}


# ------------------------------------------------------------------------------------- plainly

def _counts(x, cols, case):
    """Rows of x [cols, rows] that follow the column series: rising, falling, either."""
    L = len(cols)
    t = -(-case["num"] * (L - 1) // case["den"])
    v = x[cols]
    ge = (lambda a, b: a >= b) if case["ties"] else (lambda a, b: a > b)
    if not case["kept"]:
        inc, dec = ge(v[1:], v[:-1]).sum(0), ge(v[:-1], v[1:]).sum(0)
    else:
        inc = torch.zeros(x.shape[1], dtype=torch.int64, device=x.device)
        dec, up, down = inc.clone(), v[0].clone(), v[0].clone()
        for k in range(1, L):
            a, b = ge(v[k], up), ge(down, v[k])
            inc += a
            dec += b
            up, down = torch.where(a, v[k], up), torch.where(b, v[k], down)
    pos, neg = inc >= t, (dec >= t) & bool(case["neg"])
    return torch.stack([pos.sum(), neg.sum(), (pos | neg).sum()])


def exact(case, seed):
    if case["kind"] not in ("sweep", "noalloc", "pairs"):
        return None
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    x = _matrix(case, g).double().t().contiguous()
    if case["kind"] == "pairs":
        C = case["cols"]
        gt = torch.stack([(x > x[a]).sum(1) for a in range(C)])  # [a, b]: rows with b above a
        return torch.triu(gt + (gt.t() << 32), 1)
    col_idx, offsets = _population(case, g)
    off = offsets.tolist()
    col_idx = col_idx.long()
    p = ebic.Params.make()
    c = torch.stack([_counts(x, col_idx[a:b], case) for a, b in zip(off, off[1:])]).cpu()
    lens = torch.tensor([b - a for a, b in zip(off, off[1:])])
    fit = torch.where(c[:, 2] < p.min_rows, torch.zeros_like(lens),
                      c[:, 2] << lens.clamp(max=p.col_cap))
    return c[:, 0].int(), c[:, 1].int(), c[:, 2].int(), fit
