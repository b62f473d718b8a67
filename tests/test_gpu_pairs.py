"""Products of (hi | lo) pairs on the tensor cores, and the kernels around them, at the sizes where they can go wrong, against
the oracle: fp32 mode as pairs of fp16 words (chosen by the work of the products), bf16 pairs of metric learning and sparse
coding.  Tolerances are those of the precision modes: an fp32 value as fp16 pairs keeps 23 of its 24 bits, and the sums are
fp32, so the bound of the FMA kernels stands."""
import numpy as np
import pytest

import paper_1409_5705_b200 as S
import sfb_inputs as I
from oracle import sdca_oracle as D
from oracle import sfb_oracle as O
from _parity import TOL, config_for, oracle_step, rel_err, step_tol, to_dev

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

FP32, BF16 = pytest.param(S.PREC_FP32, id="fp32"), pytest.param(S.PREC_BF16, id="bf16")


def workload(name, rows, cols, P, B, **kw):
    base = {"mlr": dict(w_std=0.05, x_scale="unit", eta=0.05), "dml": dict(eta=1e-3), "sc": dict(eta=1e-2, sc_nnz=6)}[name]
    return I.scaled(I.WORKLOADS["mlr_mid" if name == "mlr" else name], f"{name}_pairs", rows=rows, cols=cols, workers=P, batch=B,
                    **{**base, **kw})


def check(wl, prec, per_worker=False, scale=1.0, L=None):
    W0 = (I.initial_W(wl) * np.float32(scale)).astype(np.float32)
    inp = I.step_inputs(wl, 1, I.sc_true_dictionary(wl) if wl.model == I.SC else None)
    if wl.model == I.DML:
        assert O.dml_hinge_distance(W0, inp.X, inp.Y, inp.labels) > 1e-4          # no pair on the kink: one answer
    if L is None:
        L = float(np.float32(O.lipschitz_power_iteration(W0))) if wl.model == I.SC else 0.0
    W = to_dev(W0, torch)
    ctx = S.Context(config_for(wl, prec, L), W)
    X, Y, lab = to_dev(inp.X, torch), to_dev(inp.Y, torch), to_dev(inp.labels, torch)
    if per_worker:
        for p in reversed(range(wl.workers)):
            r = slice(p * wl.batch, (p + 1) * wl.batch)
            ctx.sfb_compute_factors(p, X[r], None if Y is None else Y[r], None if lab is None else lab[r])
        ctx.sfb_gather_factors()
        ctx.sfb_apply_update()
    else:
        ctx.sfb_step(X, Y, lab)
    assert ctx.sfb_get_status() == 0
    Wg = W.cpu().numpy()
    ctx.close()
    ref = oracle_step(wl, W0, inp, L=L if wl.model == I.SC else None)
    err, tol = rel_err(Wg, ref, W0), step_tol(wl, prec, ref, W0)
    print(f"{wl.name} {wl.rows} x {wl.cols} K={wl.K}: rel err {err:.3e} (tol {tol:.3e})")
    assert err <= tol


# Ragged tiles of 256 x bn; the two forms of the update (384 and 385 pairs); rows of 2048 and 2052 columns (one warp or a block with
# bulk copies per row) and of 26,628 (registers, the rest from memory); an update of several tiles per pair of CTAs.
@pytest.mark.parametrize("shape", [(701, 1028, 3, 101), (530, 1000, 1, 384), (530, 1000, 5, 77), (640, 2048, 2, 90), (641, 2052, 2, 90),
                                   (65, 26628, 2, 70), (9001, 256, 1, 257)])
def test_regression_in_fp32(shape):
    check(workload("mlr", *shape), S.PREC_FP32)


@pytest.mark.parametrize("prec", [FP32, BF16])
@pytest.mark.parametrize("shape", [(257, 2500, 2, 193), (711, 1020, 6, 57), (64, 26628, 2, 70)])
def test_metric_learning(shape, prec):
    check(workload("dml", *shape), prec, scale=0.06)


# With and without the Gram matrix (by iterations and shape), no / one / an odd and an even number of iterations, an odd number of
# features (no 16-byte rows), more atoms than features, contractions cut over the CTA pairs.
@pytest.mark.parametrize("prec", [FP32, BF16])
@pytest.mark.parametrize("shape,iters", [((700, 400, 3, 341), 5), ((700, 400, 3, 341), 4), ((1501, 1400, 3, 47), 3), ((500, 1400, 2, 205), 4),
                                         ((257, 1092, 5, 211), 1), ((257, 1092, 5, 211), 0)])
def test_sparse_coding(shape, iters, prec):
    check(workload("sc", *shape, sc_iters=iters), prec)


# Products of more tiles than pairs of CTAs (74): at 256 columns, the widest, already ceil(K / 256) x ceil(columns / 256) of them, with the
# logits, the residual, both forms of an iteration and the first iterate.  (The coder on W^T W: bf16 mode, no more atoms than features.)
@pytest.mark.parametrize("name,shape,prec,kw", [("mlr", (5200, 516, 2, 512), S.PREC_FP32, {}), ("dml", (5200, 516, 2, 512), S.PREC_BF16, {}),
                                                ("sc", (2700, 2600, 8, 232), S.PREC_BF16, {"sc_iters": 4}),
                                                ("sc", (2564, 2700, 8, 232), S.PREC_BF16, {"sc_iters": 3}),
                                                ("sc", (2564, 2600, 8, 232), S.PREC_FP32, {"sc_iters": 3})])
def test_several_tiles_per_pair(name, shape, prec, kw):
    assert -(-shape[2] * shape[3] // 256) * -(-min(shape[:2] if name == "sc" else shape[:1]) // 256) > 74
    check(workload(name, *shape, **kw), prec, scale=0.06 if name == "dml" else 1.0)


@pytest.mark.parametrize("name,shape", [("mlr", (701, 1028, 3, 101)), ("dml", (711, 1020, 6, 57)), ("sc", (700, 400, 3, 341))])
def test_slices_of_workers_in_fp32(name, shape):
    check(workload(name, *shape, **({"sc_iters": 5} if name == "sc" else {})), S.PREC_FP32, per_worker=True, scale=0.06 if name == "dml" else 1.0)


def test_rows_of_zeros_and_wide_ranges_keep_their_scales():
    """Zero rows of W and zero samples take no part in the common scales; columns 2^16 apart keep the fp32 accuracy."""
    wl = workload("mlr", 530, 1000, 1, 400)
    rng = np.random.default_rng(3)
    col = np.exp2(np.round(np.linspace(-8, 8, wl.cols))).astype(np.float32)
    W0 = (rng.standard_normal((wl.rows, wl.cols)) * 0.02 / col).astype(np.float32)
    X = (rng.standard_normal((wl.K, wl.cols)) * col / 30).astype(np.float32)
    W0[7] = 0
    X[3] = 0
    lab = rng.integers(0, wl.rows, wl.K).astype(np.int32)
    W = to_dev(W0, torch)
    ctx = S.Context(config_for(wl, S.PREC_FP32), W)
    ctx.sfb_step(to_dev(X, torch), None, to_dev(lab, torch))
    assert ctx.sfb_get_status() == 0
    ctx.close()
    ref = O.sfb_step(wl.model, W0, X, None, lab, workers=1, eta=wl.eta)
    upd, half_ulp = np.abs(ref - W0), 0.5 * np.spacing(np.abs(ref).astype(np.float32)).astype(np.float64)
    excess = np.maximum(np.abs(W.cpu().numpy().astype(np.float64) - ref) - half_ulp, 0)
    assert (np.linalg.norm(excess, axis=0) <= TOL[S.PREC_FP32] * np.linalg.norm(upd, axis=0)).all()      # column by column


# Contractions of the logits of several k-blocks cut over the CTAs of a cluster, with tails on every side.  Operands rounded to bf16
# (about 0.8e-3 rms each) move a logit of standard deviation s by 1.15e-3 s and the factors by as much, relatively: w_std keeps s
# below 0.8 (with 0.05 it is 3.5 at 5,000 features, 4e-3, whatever the kernel does).
@pytest.mark.parametrize("shape", [(300, 4100, 2, 20), (65, 5000, 1, 129)])
def test_cut_contractions_in_bf16(shape):
    check(workload("mlr", *shape, w_std=0.01), S.PREC_BF16)


# FMA kernels: both tile sizes, contractions in parts, one and several tiles; with the Gram matrix and without.
@pytest.mark.parametrize("name,shape,kw", [("mlr", (129, 132, 1, 65), {}), ("mlr", (1000, 68, 2, 70), {}), ("mlr", (40, 3000, 1, 33), {}),
                                           ("dml", (130, 1000, 2, 70), {}), ("sc", (260, 132, 2, 70), {"sc_iters": 4}),
                                           ("sc", (101, 260, 1, 5), {"sc_iters": 3})])
def test_fma_products(name, shape, kw):
    check(workload(name, *shape, **kw), S.PREC_FP32_FFMA, scale=0.06 if name == "dml" else 1.0)


# The estimate of L: on W^T W (fewer rows than blocks, rows of G in shared memory and beyond it) and on W with the vector in shared
# memory and beyond it.  50 products of fp32 sums: 50 * 2^-24 of L, and in bf16 mode W itself to 2^-17.
@pytest.mark.parametrize("rows,cols,K,prec", [(21, 4, 64, S.PREC_FP32), (162, 208, 308, S.PREC_FP32), (2000, 1000, 128, S.PREC_FP32),
                                              (300, 3000, 64, S.PREC_BF16), (100, 60000, 4, S.PREC_FP32), (2685, 1952, 30, S.PREC_BF16)])
def test_lipschitz_estimate(rows, cols, K, prec):
    wl = workload("sc", rows, cols, 1, K, sc_iters=2)
    W0 = I.initial_W(wl)
    X = np.random.default_rng(5).standard_normal((K, rows)).astype(np.float32)
    W = to_dev(W0, torch)
    ctx = S.Context(config_for(wl, prec, 0.0, prox=0), W)
    ctx.sfb_step(to_dev(X, torch), None, None)
    assert ctx.sfb_get_status() == 0
    L = ctx.sfb_get_stats().sc_lipschitz
    ctx.close()
    ref = O.lipschitz_power_iteration(W0)
    assert abs(L - ref) <= (50 * 2.0 ** -24 if prec == S.PREC_FP32 else 2.0 ** -16) * ref


# The forward product of sparse samples on the FMA kernels: over the scattered samples (few columns) and row by row (many).
@pytest.mark.parametrize("rows,cols,P,B,nnz", [(3000, 148, 2, 40, 13), (500, 20000, 2, 16, 30)])
def test_sparse_samples_in_fp32(rows, cols, P, B, nnz):
    wl = workload("mlr", rows, cols, P, B)
    W0 = I.initial_W(wl)
    sp = I.sparse_samples(wl.seed, 1, wl.K, cols, float(nnz))
    lab = I.zipf_labels(wl.seed, 5, 1, wl.K, rows, wl.zipf_s)
    W = to_dev(W0, torch)
    ctx = S.Context(S.make_config(wl.model, rows, cols, P, B, wl.eta, S.PREC_FP32_FFMA, csr_nnz_max=sp.nnz), W)
    ctx.sfb_step_csr(to_dev(sp.indptr, torch), to_dev(sp.indices, torch), to_dev(sp.values, torch), sp.nnz, to_dev(lab, torch))
    assert ctx.sfb_get_status() == 0
    ref = O.sfb_step(wl.model, W0, I.densify(sp, cols), None, lab, workers=P, eta=wl.eta)
    err = rel_err(W.cpu().numpy(), ref, W0)
    ctx.close()
    assert err <= TOL[S.PREC_FP32]


# The dual solve with the scores of a sample in shared memory (up to 51,200 classes) and re-read.
@pytest.mark.parametrize("classes", [51200, 51204])
def test_dual_solve_at_the_edge_of_shared_memory(classes):
    N, dim, P, B, lam = 12, 8, 1, 3, 0.1
    A = (I.normal_matrix(0, 31, N, dim, 1.0) * np.float32(3.0 / np.sqrt(dim))).astype(np.float32)
    y = (np.arange(N) * 977 % classes).astype(np.int32)
    W = torch.zeros((classes, dim), dtype=torch.float32, device="cuda")
    Q = to_dev(D.initial_dual(y, classes).astype(np.float32), torch)
    ctx = S.Context(S.make_config(S.L2MLR, classes, dim, P, B, 1.0 / 3, S.PREC_FP32, sdca_lambda=lam, sdca_n=N), W)
    ctx.sfb_sdca_set_dual(Q)
    for step in range(2):
        ids = np.array([1, 5, 9], dtype=np.int32) + step
        W_t, Q_t = W.cpu().numpy(), Q.cpu().numpy()
        ctx.sfb_sdca_step(to_dev(A[ids], torch), to_dev(y[ids], torch), to_dev(ids, torch))
        assert ctx.sfb_get_status() == 0
        W_ref, Q_ref, _, _ = D.sdca_step(W_t, A[ids], y[ids], ids, Q_t, lam, 1.0 / 3, workers=P)
        err = np.linalg.norm(W.cpu().numpy().astype(np.float64) - W_ref.astype(np.float32)) / np.linalg.norm(W_ref - W_t)
        assert err <= TOL[S.PREC_FP32] and np.abs(Q.cpu().numpy() - Q_ref).max() <= 2e-6
    ctx.close()


# Samples from host memory: copied in parts beside the products of the parts before them (several times 128 samples), in one piece.
@pytest.mark.parametrize("shape", [(2000, 8000, 4, 64), (1000, 8000, 1, 384), (333, 260, 3, 37)])
def test_host_samples_in_parts(shape):
    # (samples of unit length: of 8,000 unit features, length 90, one step puts every p_y at 1 and leaves a second update of 0)
    wl = workload("mlr", *shape, w_std=0.01, x_scale="inv_sqrt_d")
    W0, inp = I.initial_W(wl), I.step_inputs(wl, 1)
    W = to_dev(W0, torch)
    ctx = S.Context(config_for(wl, S.PREC_BF16), W)
    X, lab = torch.from_numpy(inp.X).pin_memory(), torch.from_numpy(inp.labels).pin_memory()
    Wt = W0
    for _ in range(2):                                          # the second step copies over the first one's samples
        loss, status = ctx.sfb_step_host(X, None, lab)
        ref, Wg = oracle_step(wl, Wt, inp), W.cpu().numpy()
        assert status == 0 and abs(loss - O.mlr_loss(Wt, inp.X, inp.labels).mean()) < 1e-3
        assert rel_err(Wg, ref, Wt) <= TOL[S.PREC_BF16]
        Wt = Wg
    ctx.close()
