"""Inputs at the ends of the ranges that the entry points take, and calls in orders that a program may use them in: workspace
memory with anything in it, matrices of large and small norm, W written between two calls, steps in which a coder does not
converge."""
import numpy as np
import pytest

import paper_1409_5705_b200 as S
import sfb_inputs as I
from oracle import sfb_oracle as O
from _parity import config_for, oracle_step, rel_err, step_tol, to_dev

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def poisoned_context(cfg, W, monkeypatch):
    """A context whose workspace holds NaN in every word at the start."""
    empty = torch.empty
    with monkeypatch.context() as m:
        m.setattr(torch, "empty", lambda *a, **k: empty(*a, **k).fill_(255) if k.get("dtype") is torch.uint8 else empty(*a, **k))
        return S.Context(cfg, W)


def sc_workload(rows, cols, K, iters, **kw):
    return I.scaled(I.WORKLOADS["sc"], "sc_ranges", rows=rows, cols=cols, workers=1, batch=K, eta=1e-2, sc_nnz=6, sc_iters=iters, **kw)


# rows % 4 = 0 .. 3: what lies between `rows` and the pitch of u must not reach the products of the next step.
@pytest.mark.parametrize("rows", [1500, 1501, 1502, 1503])
@pytest.mark.parametrize("prec", [pytest.param(S.PREC_FP32, id="fp32"), pytest.param(S.PREC_BF16, id="bf16")])
def test_second_step_on_a_workspace_of_nan(rows, prec, monkeypatch):
    wl = sc_workload(rows, 600, 400, 3)
    W0 = I.initial_W(wl)
    L = float(np.float32(O.lipschitz_power_iteration(W0)))
    W = to_dev(W0, torch)
    ctx = poisoned_context(config_for(wl, prec, L), W, monkeypatch)
    Wt, D = W0, I.sc_true_dictionary(wl)
    for t in range(2):
        inp = I.step_inputs(wl, t, D)
        ctx.sfb_step(to_dev(inp.X, torch), None, None)
        assert ctx.sfb_get_status() == 0
        Wg, ref = W.cpu().numpy(), oracle_step(wl, Wt, inp, L=L)
        assert rel_err(Wg, ref, Wt) <= step_tol(wl, prec, ref, Wt)
        Wt = Wg
    ctx.close()


# The estimate of L on W^T W, on W with the vector in shared memory, and beyond it (51,200 atoms), for dictionaries of any norm: the
# lengths of the iterates must neither overflow nor vanish.  50 products of fp32 sums: 50 * 2^-24 of L.
@pytest.mark.parametrize("scale", [1e-8, 1e-4, 1.0, 3e3, 1e5, 1e8])
@pytest.mark.parametrize("rows,cols,K", [(400, 200, 64), (60, 700, 2), (40, 60000, 2)])
def test_lipschitz_estimate_of_small_and_large_dictionaries(rows, cols, K, scale):
    wl = sc_workload(rows, cols, K, 2)
    W0 = (I.initial_W(wl) * np.float32(scale)).astype(np.float32)
    X = np.random.default_rng(5).standard_normal((K, rows)).astype(np.float32)
    W = to_dev(W0, torch)
    ctx = S.Context(config_for(wl, S.PREC_FP32, 0.0, prox=0), W)
    ctx.sfb_step(to_dev(X, torch), None, None)
    assert ctx.sfb_get_status() == 0
    L = ctx.sfb_get_stats().sc_lipschitz
    ctx.close()
    ref = O.lipschitz_power_iteration(W0)
    assert abs(L - ref) <= 50 * 2.0 ** -24 * ref


# Factors that are computed again before any update, after the caller has written W (a line search, a check of gradients): they
# belong to the W of the second call, on every kind of kernel.  all: one call for all workers; else worker 0 again.
@pytest.mark.parametrize("whole", [True, False])
@pytest.mark.parametrize("model,shape,prec", [(S.MLR, (701, 1028, 2, 180), S.PREC_FP32), (S.MLR, (70, 260, 2, 20), S.PREC_FP32),
                                              (S.DML, (300, 2500, 2, 150), S.PREC_FP32), (S.DML, (300, 2500, 2, 150), S.PREC_BF16),
                                              (S.SC, (700, 400, 2, 512), S.PREC_FP32), (S.SC, (260, 132, 2, 40), S.PREC_FP32)])
def test_factors_computed_again_see_the_w_of_now(model, shape, prec, whole):
    rows, cols, P, B = shape
    rng = np.random.default_rng(2)
    K, ind = P * B, rows if model == S.SC else cols
    W0 = (rng.standard_normal((rows, cols)) / np.sqrt(rows if model == S.SC else cols)).astype(np.float32)
    X, Y = (rng.standard_normal((K, ind)).astype(np.float32) for _ in range(2))
    lab = rng.integers(0, rows if model == S.MLR else 2, K).astype(np.int32)
    W = to_dev(W0, torch)
    cfg = S.make_config(model, rows, cols, P, B, 1e-3, prec, sc_ista_iters=4)
    ctx = S.Context(cfg, W)
    dev = [to_dev(a, torch) for a in (X, Y if model == S.DML else None, lab if model != S.SC else None)]
    part = dev if whole else [None if a is None else a[:B] for a in dev]
    ctx.sfb_compute_factors(-1, *dev)
    W.mul_(0.5)
    ctx.sfb_compute_factors(-1 if whole else 0, *part)
    U, V = (t.cpu().numpy().astype(np.float64) for t in ctx.factors_as_tensors())
    ctx.close()
    n, Wn = K if whole else B, (W0 * np.float32(0.5)).astype(np.float64)
    L = O.lipschitz_power_iteration(Wn.astype(np.float32)) if model == S.SC else None
    Ur, Vr = O.sfb_step(model, Wn, X, Y, lab, workers=P, eta=1e-3, margin=1.0, lam=0.1, L=L, iters=4, prox=False, return_factors=True)[1:3]
    for got, want in ((U[:n], Ur[:n]), (V[:n], Vr[:n])):
        assert np.linalg.norm(got - want) <= (1e-5 if prec == S.PREC_FP32 else 1e-4) * np.linalg.norm(want)


# Codes and residuals of samples that the dictionary fits, 20 iterations in fp32 mode, on every form of the coder: W^T W in fp64 (tiles of
# 64 with remainders, odd slices of samples, contractions in parts), two products on the FMA kernels, pairs of fp16 words.  The
# gradient cancels, so this shows what the norm of W after a step does not: an error of 2^-24 of W^T W a instead of the residual
# gave 2e-6 for the codes and 1e-5 for the residual.  Bounds: 10 * 2^-24 of the codes, and of x for W a - x.
@pytest.mark.parametrize("rows,cols,P,B", [(1404, 296, 1, 742), (772, 1280, 2, 467), (2000, 1000, 1, 128), (301, 200, 3, 11), (1, 4, 1, 1), (90, 64, 1, 65),
                                           (2100, 68, 1, 5), (150, 1104, 1, 9), (700, 132, 2, 97)])
def test_codes_of_fitted_samples(rows, cols, P, B):
    rng = np.random.default_rng(rows + cols)
    W0 = rng.standard_normal((rows, cols)).astype(np.float32)
    W0 /= np.linalg.norm(W0, axis=0, keepdims=True)
    K, nz = P * B, min(20, cols)
    a = np.zeros((K, cols))
    for i in range(K):
        a[i, rng.choice(cols, nz, replace=False)] = rng.standard_normal(nz)
    X = (a @ W0.T.astype(np.float64) + 0.01 * rng.standard_normal((K, rows))).astype(np.float32)
    Wd = W0.astype(np.float64)
    L = float(np.float32(np.linalg.norm(Wd, 2) ** 2 * 1.01))
    W = to_dev(W0, torch)
    ctx = S.Context(S.make_config(S.SC, rows, cols, P, B, 1e-3, S.PREC_FP32, sc_lambda=0.1, sc_ista_iters=20, sc_lipschitz=L), W)
    Xd = to_dev(X, torch)
    for p in range(P):
        ctx.sfb_compute_factors(p, Xd[p * B:(p + 1) * B].clone())
    U, V = (t.cpu().numpy().astype(np.float64) for t in ctx.factors_as_tensors())
    assert ctx.sfb_get_status() == 0
    ctx.close()
    c = np.zeros((K, cols))
    for _ in range(20):
        g = c - (c @ Wd.T - X) @ Wd / L
        c = np.sign(g) * np.maximum(np.abs(g) - 0.1 / L, 0)
    assert np.linalg.norm(V - c) <= 10 * 2.0 ** -24 * np.linalg.norm(c)
    assert np.linalg.norm(U - (c @ Wd.T - X)) <= 10 * 2.0 ** -24 * np.linalg.norm(X)


# An L below ||W||^2 / 2, on which the iterations diverge (values of 1e8 and more here): still the iterates, to the precision of the mode, on
# pairs of words with scales, in fp64 and on the FMA kernels.
@pytest.mark.parametrize("rows,cols,P,B,T", [(772, 1280, 2, 467, 20), (772, 1280, 2, 467, 7), (2000, 1000, 1, 128, 20), (2000, 1400, 4, 128, 20), (90, 64, 1, 8, 12)])
def test_codes_of_diverging_iterations(rows, cols, P, B, T):
    rng = np.random.default_rng(rows + cols)
    W0 = rng.standard_normal((rows, cols)).astype(np.float32)
    W0 /= np.linalg.norm(W0, axis=0, keepdims=True)
    K = P * B
    X = rng.standard_normal((K, rows)).astype(np.float32)
    X[1] *= 1e-3
    Wd = W0.astype(np.float64)
    L = float(np.float32(np.linalg.norm(Wd, 2) ** 2 / 6))
    W = to_dev(W0, torch)
    ctx = S.Context(S.make_config(S.SC, rows, cols, P, B, 1e-3, S.PREC_FP32, sc_lambda=0.1, sc_ista_iters=T, sc_lipschitz=L), W)
    ctx.sfb_compute_factors(-1, to_dev(X, torch))
    U, V = (t.cpu().numpy().astype(np.float64) for t in ctx.factors_as_tensors())
    assert ctx.sfb_get_status() == 0
    ctx.close()
    c = np.zeros((K, cols))
    for _ in range(T):
        g = c - (c @ Wd.T - X) @ Wd / L
        c = np.sign(g) * np.maximum(np.abs(g) - 0.1 / L, 0)
    assert np.linalg.norm(V - c) <= 1e-5 * np.linalg.norm(c)
    u = c @ Wd.T - X
    assert np.linalg.norm(U - u) <= 1e-5 * np.linalg.norm(u)


# More than 65,535 blocks of 64 features.
@pytest.mark.parametrize("prec", [pytest.param(S.PREC_FP32, id="fp32"), pytest.param(S.PREC_BF16, id="bf16")])
def test_sparse_coding_of_millions_of_features(prec):
    rows, cols, K, T = 4_194_400, 64, 128, 3
    g = torch.Generator(device="cuda").manual_seed(1)
    W = torch.randn(rows, cols, generator=g, device="cuda") / np.sqrt(rows)
    X = torch.randn(K, rows, generator=g, device="cuda") / np.sqrt(rows) + torch.randn(K, cols, generator=g, device="cuda") @ W.t()
    Wd, Xd, L = W.double(), X.double(), 1.1
    c = torch.zeros(K, cols, dtype=torch.float64, device="cuda")
    for _ in range(T):
        a = c - (c @ Wd.t() - Xd) @ Wd / L
        c = torch.sign(a) * (a.abs() - 0.1 / L).clamp_min(0)
    ctx = S.Context(S.make_config(S.SC, rows, cols, 1, K, 1e-3, prec, sc_lambda=0.1, sc_ista_iters=T, sc_lipschitz=L), W)
    ctx.sfb_compute_factors(-1, X)
    V = ctx.factors_as_tensors()[1]
    assert ctx.sfb_get_status() == 0
    ctx.close()
    assert float((V.double() - c).norm()) <= (1e-5 if prec == S.PREC_FP32 else 1e-4) * float(c.norm())


# The loss of a step can be read after the gather, before the update.
@pytest.mark.parametrize("prec", [pytest.param(S.PREC_FP32, id="fp32"), pytest.param(S.PREC_BF16, id="bf16")])
def test_loss_after_the_gather(prec):
    wl = I.scaled(I.WORKLOADS["mlr_mid"], "loss", rows=333, cols=260, workers=3, batch=37, eta=0.05, w_std=0.05, x_scale="unit")
    W0 = I.initial_W(wl)
    W = to_dev(W0, torch)
    ctx = S.Context(config_for(wl, prec), W)
    Wt = W0
    for t in range(3):
        inp = I.step_inputs(wl, t)
        X, lab = to_dev(inp.X, torch), to_dev(inp.labels, torch)
        for p in range(wl.workers):
            r = slice(p * wl.batch, (p + 1) * wl.batch)
            ctx.sfb_compute_factors(p, X[r], None, lab[r])
        ctx.sfb_gather_factors()
        if t:                                                    # (the read-outs begin with the first completed step)
            assert abs(ctx.sfb_get_stats().last_loss - O.mlr_loss(Wt, inp.X, inp.labels).mean()) < 2e-3
        ctx.sfb_apply_update()
        Wt = W.cpu().numpy()
        assert abs(ctx.sfb_get_stats().last_loss - O.mlr_loss(I.initial_W(wl) if t == 0 else Wprev, inp.X, inp.labels).mean()) < 2e-3
        Wprev = Wt
    ctx.close()


# A context with room for sparse samples whose products of dense samples belong on the tensor cores and those of sparse ones on the FMA
# kernels: dense, sparse and mixed steps in turn on one context, factors received and an update replayed between them.
def test_dense_and_sparse_steps_on_one_fp32_context():
    rows, cols, P, B = 2000, 4000, 4, 32
    wl = I.scaled(I.WORKLOADS["mlr_mid"], "mixed", rows=rows, cols=cols, workers=P, batch=B, eta=0.05, w_std=0.01, x_scale="inv_sqrt_d")
    W0 = I.initial_W(wl)
    W = to_dev(W0, torch)
    ctx = S.Context(S.make_config(S.MLR, rows, cols, P, B, wl.eta, S.PREC_FP32, csr_nnz_max=8 * wl.K * 2), W)
    Wt, flops = W0, []
    for t, form in enumerate(["dense", "sparse", "dense", "mixed", "sparse", "received", "mixed", "dense"]):
        inp = I.step_inputs(wl, t)
        sp = I.sparse_samples(wl.seed, t, wl.K, cols, 8.0)
        X, lab = inp.X.copy(), inp.labels
        ld = to_dev(lab, torch)
        before = ctx.sfb_get_stats().flops
        if form == "dense":
            ctx.sfb_step(to_dev(X, torch), None, ld)
        elif form == "sparse":
            X = I.densify(sp, cols)
            ctx.sfb_step_csr(to_dev(sp.indptr, torch), to_dev(sp.indices, torch), to_dev(sp.values, torch), sp.nnz, ld)
        else:
            for p in range(P):
                r = slice(p * B, (p + 1) * B)
                if p % 2 == 0:
                    X[r] = I.densify(sp, cols)[r]
                    ip = sp.indptr[p * B:(p + 1) * B + 1]
                    lo, hi = int(ip[0]), int(ip[-1])
                    ctx.sfb_compute_factors_csr(p, to_dev(ip - lo, torch), to_dev(sp.indices[lo:hi], torch), to_dev(sp.values[lo:hi], torch), hi - lo, ld[r])
                else:
                    ctx.sfb_compute_factors(p, to_dev(X[r], torch), None, ld[r])
                if form == "received" and p != 1:
                    U, V = torch.empty(B, rows, device="cuda"), torch.empty(B, cols, device="cuda")
                    ctx.sfb_export_factors(p, U, V)
                    ctx.sfb_set_factors(p, U, V)
            ctx.sfb_gather_factors()
            ctx.sfb_apply_update()
        assert ctx.sfb_get_status() == 0
        flops.append(ctx.sfb_get_stats().flops - before)
        Wg, ref = W.cpu().numpy(), O.sfb_step(wl.model, Wt, X, None, lab, workers=P, eta=wl.eta)
        assert rel_err(Wg, ref, Wt) <= 1e-5, form
        if t == 3 or t == 5:
            ctx.sfb_replay_update()
            assert rel_err(W.cpu().numpy(), Wg.astype(np.float64) + (ref - Wt), Wt) <= 2e-5, form
            Wg = W.cpu().numpy()
        Wt = Wg
    ctx.close()
    assert flops[0] >= 7.5 * wl.K * rows * cols                   # three products a term in the logits of dense samples


# Which update a step of sparse samples takes in bf16 mode: from 200,000 rows on the sparse one again, below one non-zero per column.
@pytest.mark.parametrize("rows,sparse", [(200_000, True), (199_999, False)])
def test_choice_of_the_update_by_rows(rows, sparse):
    cols, K = 2048, 1024
    sp = I.sparse_samples(3, 0, K, cols, 0.4)                     # one entry a sample
    lab = np.arange(K, dtype=np.int32)
    W = torch.zeros((rows, cols), device="cuda")
    ctx = S.Context(S.make_config(S.MLR, rows, cols, 16, 64, 0.05, S.PREC_BF16, csr_nnz_max=sp.nnz), W)
    ctx.sfb_step_csr(to_dev(sp.indptr, torch), to_dev(sp.indices, torch), to_dev(sp.values, torch), sp.nnz, to_dev(lab, torch))
    assert ctx.sfb_get_status() == 0 and ctx.sfb_get_stats().sparse_updates == int(sparse)
    ctx.close()
