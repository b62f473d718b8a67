"""The work that users of this library have it do, as cases that can be timed and compared.

A case is one minibatch step through the public entry points of ``paper_1409_5705_b200``: multiclass logistic regression
("mlr"), distance metric learning ("dml"), sparse coding ("sc") and l2-regularised logistic regression by dual ascent
("l2mlr"), in the tensor-core (bf16) and the fp32 operand precision, from the smallest workload of the repository to its
paper-scale one.  ``form`` says how the program makes the step:

  step     all K = workers x batch samples resident on the device, one call
  workers  one factors call per logical worker, then gather and update (the loop of the paper)
  host     samples in pinned host memory, one call that copies them in and returns the loss and the status word
  csr      samples in compressed-sparse-row form on the device

A state holds four minibatches that the passes take in turn, as a training loop does; every pass moves W.
"""
import math

import torch

import paper_1409_5705_b200 as S

_MODEL = {"mlr": S.MLR, "dml": S.DML, "sc": S.SC, "l2mlr": S.L2MLR}
_PREC = {"bf16": S.PREC_BF16, "fp32": S.PREC_FP32}
_BATCHES = 4
_ETA = {"mlr": 0.05, "dml": 1e-3, "sc": 1e-3}
_LAMBDA = 0.1                      # l1 weight of the sparse coder; regulariser of l2mlr
_PROX_WEIGHT = 1e-4                # l1 weight of the entry-wise prox, where a case has it


def _case(name, model, prec, rows, cols, workers, batch, form="step", nnz=0, prox=False, estimate=False, zero=False):
    """nnz: mean non-zeros per sample (csr); prox: entry-wise l1 prox in the update; estimate: the library estimates the
    coder's step size every step instead of being given it; zero: training starts at W = 0 with unscaled features."""
    return {"name": name, "model": model, "prec": prec, "rows": rows, "cols": cols, "workers": workers, "batch": batch,
            "form": form, "nnz": nnz, "prox": prox, "estimate": estimate, "zero": zero}


def listed():
    return [
        # the smallest workload of the repository: a few microseconds of work, so launches and host time are what a user sees
        _case("mlr_tiny_bf16", "mlr", "bf16", 64, 256, 4, 32, zero=True),
        # ten thousand classes, twenty thousand features: the ordinary training step, in the default fast precision ...
        _case("mlr_mid_bf16", "mlr", "bf16", 10_000, 20_000, 16, 64),
        # ... and in the 1e-5 precision, for users who need fp32 operands
        _case("mlr_mid_fp32", "mlr", "fp32", 10_000, 20_000, 16, 64),
        # the paper-scale matrix (13 GB), the repository's default benchmark
        _case("mlr_large_bf16", "mlr", "bf16", 325_000, 10_000, 16, 64),
        # odd sizes, every worker's factors computed by a call of its own, with an l1 penalty on W
        _case("mlr_ragged_workers_bf16", "mlr", "bf16", 4_999, 3_004, 7, 37, form="workers", prox=True),
        # minibatches that come from a loader in host memory; the loss is read every step
        _case("mlr_host_bf16", "mlr", "bf16", 20_000, 4_000, 8, 64, form="host"),
        # metric learning at the size of the repository's workload, in both precisions
        _case("dml_bf16", "dml", "bf16", 1_000, 20_000, 16, 64),
        _case("dml_fp32", "dml", "fp32", 1_000, 20_000, 16, 64),
        # dictionary learning at the size of the repository's workload: twenty coder iterations, column prox
        _case("sc_bf16", "sc", "bf16", 10_000, 5_000, 16, 32),
        # a small dictionary in fp32, the coder's step size left to the library
        _case("sc_small_fp32", "sc", "fp32", 2_000, 1_000, 8, 16, estimate=True),
        # tf-idf-like sparse samples against the ordinary matrix
        _case("mlr_csr_bf16", "mlr", "bf16", 10_000, 20_000, 16, 64, form="csr", nnz=30),
        # dual ascent for the l2-regularised model
        _case("l2mlr_bf16", "l2mlr", "bf16", 10_000, 4_000, 8, 64),
    ]


def _cost(c):
    """Multiply-adds of a step times what one costs relative to a bf16 tensor-core product at the same size."""
    mac = float(c["workers"] * c["batch"]) * c["rows"] * c["cols"]
    passes = 42.0 if c["model"] == "sc" else 2.0
    big = c["model"] in ("mlr", "l2mlr") and c["rows"] >= 2048 and c["cols"] >= 512 and c["workers"] * c["batch"] >= 128
    weight = (6.0 if big else 25.0) if c["prec"] == "fp32" else 1.0 if c["model"] in ("mlr", "l2mlr") else 4.0
    return mac * passes * weight


_MOST = 2.0 * 1024 * 325_000 * 10_000          # the largest listed case


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["mlr/bf16/step", "mlr/bf16/step", "mlr/bf16/workers", "mlr/bf16/host", "mlr/bf16/csr",
                       "mlr/fp32/step", "mlr/fp32/workers", "mlr/fp32/csr", "dml/bf16/step", "dml/bf16/workers",
                       "dml/fp32/step", "sc/bf16/step", "sc/fp32/step", "l2mlr/bf16/step", "l2mlr/fp32/step"])
    model, prec, form = kind.split("/")
    top_rows = {"mlr": 325_000, "l2mlr": 50_000, "dml": 1_000, "sc": 10_000}[model]
    top_cols = {"mlr": 20_000, "l2mlr": 20_000, "dml": 20_000, "sc": 5_000}[model]
    if kind == "sc/fp32/step":                 # twenty coder iterations in fp32: dictionaries of moderate size
        top_rows, top_cols = 2_500, 1_500
    while True:
        c = _case("", model, prec, log_int(64, top_rows), 4 * log_int(32, top_cols // 4), rng.randint(1, 16),
                  log_int(8, 64), form=form, prox=model == "mlr" and rng.random() < 0.25,
                  estimate=model == "sc" and rng.random() < 0.5)
        if form == "csr":
            c["nnz"] = log_int(10, max(11, min(300, c["cols"] // 8)))
        if _cost(c) <= _MOST:
            del c["name"]
            return c


# ---------------------------------------------------------------------------------------------------------------------
# Inputs, drawn on the device from the seed
# ---------------------------------------------------------------------------------------------------------------------
def _zipf_labels(g, n, classes, s):
    w = torch.arange(1, classes + 1, dtype=torch.float64, device="cuda") ** (-s)
    cdf = torch.cumsum(w, 0)
    u = torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * cdf[-1]
    return torch.searchsorted(cdf, u, right=True).clamp_(max=classes - 1).to(torch.int32)


def _unit_columns(g, rows, cols):
    W = torch.randn(rows, cols, generator=g, device="cuda")
    return W.div_(W.norm(dim=0, keepdim=True))


def _sparse_rows(g, n, cols, mean):
    """tf-idf-like rows: Poisson counts, columns without replacement with Zipf(1) popularity, log-normal values, unit length."""
    rate = torch.full((n,), float(mean), device="cuda")
    counts = torch.poisson(rate, generator=g).clamp_(1, cols).long()
    rank = torch.randperm(cols, generator=g, device="cuda")
    score = -torch.log(rank + 1.0) - torch.log(-torch.log(torch.rand(n, cols, generator=g, device="cuda").clamp_(1e-12, 1 - 1e-7)))
    top = int(counts.max())
    idx = torch.topk(score, top, dim=1).indices
    keep = torch.arange(top, device="cuda")[None, :] < counts[:, None]
    idx = torch.where(keep, idx, cols).sort(dim=1).values
    val = torch.exp(0.5 * torch.randn(n, top, generator=g, device="cuda")) * keep
    val = val / val.norm(dim=1, keepdim=True)
    indptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    indptr[1:] = torch.cumsum(counts, 0)
    return indptr, idx[keep].to(torch.int32).contiguous(), val[keep].contiguous(), int(indptr[-1])


def _lipschitz(W):
    b = torch.full((W.shape[1],), W.shape[1] ** -0.5, device="cuda")
    for _ in range(50):
        b = W.t() @ (W @ b)
        b /= b.norm()
    return float((W @ b).square().sum())


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    model, rows, cols, P, B = case["model"], case["rows"], case["cols"], case["workers"], case["batch"]
    K = P * B
    more, batches, Q = {}, [], None
    if model in ("mlr", "l2mlr"):
        if case["zero"] or model == "l2mlr":
            W = torch.zeros(rows, cols, device="cuda")
        else:
            W = torch.randn(rows, cols, generator=g, device="cuda").mul_(0.01)
        scale = 1.0 if case["zero"] else (3.0 if model == "l2mlr" else 1.0) / math.sqrt(cols)
        for t in range(_BATCHES):
            y = _zipf_labels(g, K, rows, 0.0 if case["zero"] else 1.0)
            if case["form"] == "csr":
                batches.append(_sparse_rows(g, K, cols, case["nnz"]) + (y,))
            else:
                batches.append([torch.randn(K, cols, generator=g, device="cuda").mul_(scale), None, y])
        if case["form"] == "csr":
            more["csr_nnz_max"] = max(b[3] for b in batches)
        if model == "l2mlr":
            n = _BATCHES * K
            Q = torch.zeros(n, rows, device="cuda")          # u = 0: every dual row at its label's corner
            Q[torch.arange(n, device="cuda"), torch.cat([b[2] for b in batches]).long()] = 1.0
            ids = torch.randperm(n, generator=g, device="cuda")
            order = torch.argsort(ids)
            Q = Q[order].contiguous()
            for t, b in enumerate(batches):
                b[1] = ids[t * K:(t + 1) * K].to(torch.int32).contiguous()
            more.update(sdca_lambda=_LAMBDA, sdca_n=n)
    elif model == "dml":
        W = torch.randn(rows, cols, generator=g, device="cuda").mul_(1.0 / math.sqrt(cols))
        for t in range(_BATCHES):
            X = torch.randn(K, cols, generator=g, device="cuda")
            Z = torch.randn(K, cols, generator=g, device="cuda")
            same = (torch.rand(K, generator=g, device="cuda") < 0.5).to(torch.int32)
            batches.append([X, torch.where(same[:, None] == 1, X + 0.1 * Z, Z), same])
    else:
        W = _unit_columns(g, rows, cols)
        true = _unit_columns(g, rows, cols)
        nz = min(20, cols)
        for t in range(_BATCHES):
            a = torch.zeros(K, cols, device="cuda")
            at = torch.rand(K, cols, generator=g, device="cuda").topk(nz, dim=1).indices
            a.scatter_(1, at, torch.randn(K, nz, generator=g, device="cuda"))
            batches.append([a @ true.t() + 0.01 * torch.randn(K, rows, generator=g, device="cuda"), None, None])
        more.update(sc_lambda=_LAMBDA, sc_ista_iters=20, sc_prox=1, sc_lipschitz=0.0 if case["estimate"] else _lipschitz(W))
    if case["form"] == "host":
        batches = [[None if a is None else a.cpu().pin_memory() for a in b] for b in batches]
    elif case["form"] == "workers":
        cut = lambda a, p: None if a is None else a[p * B:(p + 1) * B]  # noqa: E731
        batches = [[[cut(a, p) for a in b] for p in range(P)] for b in batches]
    eta = 1.0 / K if model == "l2mlr" else 0.01 if case["zero"] else _ETA[model]
    if case["prox"]:
        more.update(prox_kind=S.PROX_L1, prox_weight=_PROX_WEIGHT)
    ctx = S.Context(S.make_config(_MODEL[model], rows, cols, P, B, eta, _PREC[case["prec"]], **more), W)
    if Q is not None:
        ctx.sfb_sdca_set_dual(Q)
    return {"ctx": ctx, "W": W, "Q": Q, "batches": batches, "next": 0, "form": "sdca" if Q is not None else case["form"]}


def run(state):
    ctx, form = state["ctx"], state["form"]
    b = state["batches"][state["next"]]
    state["next"] = (state["next"] + 1) % _BATCHES
    if form == "step":
        ctx.sfb_step(b[0], b[1], b[2])
    elif form == "workers":
        for p, (X, Y, labels) in enumerate(b):
            ctx.sfb_compute_factors(p, X, Y, labels)
        ctx.sfb_gather_factors()
        ctx.sfb_apply_update()
    elif form == "host":
        loss, status = ctx.sfb_step_host(b[0], b[1], b[2])
        return {"W": state["W"], "loss": loss, "status": status}
    elif form == "csr":
        ctx.sfb_step_csr(*b)
    else:
        ctx.sfb_sdca_step(b[0], b[2], b[1])
        return {"W": state["W"], "Q": state["Q"]}
    return state["W"]


# ---------------------------------------------------------------------------------------------------------------------
def work(case):
    """W read and written once, the samples read once; the products of the step at 2 flops per multiply-add."""
    rows, cols, K = case["rows"], case["cols"], case["workers"] * case["batch"]
    mat = float(rows) * cols
    nbytes = 8.0 * mat
    if case["form"] == "csr":
        nnz = float(K) * case["nnz"]
        return {"bytes": nbytes + 8.0 * nnz + 12.0 * K, "flops": 4.0 * nnz * rows}
    if case["model"] == "sc":
        flops = 2.0 * K * mat * 42 + (2.0 * mat * 101 if case["estimate"] else 0.0)     # 41 coder products and the update
        return {"bytes": nbytes + 4.0 * K * rows, "flops": flops}
    nbytes += 4.0 * K * cols * (2 if case["model"] == "dml" else 1) + 4.0 * K
    if case["model"] == "l2mlr":
        nbytes += 8.0 * K * rows + 4.0 * K
    return {"bytes": nbytes, "flops": 4.0 * K * mat}


def tolerance(case):
    """fp32 sums: 1e-5 of the result.  The logistic models in bf16 round their operands to 8 bits: 2e-3 of the UPDATE, which
    is the share of W that a step changes (all of it from a zero start; else about eta sqrt(K) |x| against 0.01 sqrt(rows
    cols))."""
    if case["prec"] == "fp32" or case["model"] not in ("mlr", "l2mlr"):
        return {"rel": 1e-5}
    if case["zero"] or case["model"] == "l2mlr":
        return {"rel": 2e-3}
    share = _ETA["mlr"] * math.sqrt(case["workers"] * case["batch"]) / (0.01 * math.sqrt(float(case["rows"]) * case["cols"]))
    return {"rel": max(1e-5, 2e-3 * min(1.0, 2.0 * share))}
