"""Regression in bf16 mode at the sizes where the choice of its kernels changes and their tiles end, against the oracle at the mode's
tolerance; the operand copy of W must be bf16(W) bit for bit after the step."""
import pytest

import paper_1409_5705_b200 as S
import sfb_inputs as I
from _parity import TOL, config_for, oracle_step, rel_err, to_dev

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def check(rows, cols, workers, batch, per_worker=False):
    # logits of about 1: those of size s carry 2^-9 s of rounding in bf16 operands, and the probabilities with them (with s = 4.8 the
    # update is 3.0e-3 off on any kernel)
    wl = I.scaled(I.WORKLOADS["mlr_mid"], "mlr_forms", rows=rows, cols=cols, workers=workers, batch=batch, w_std=cols ** -0.5,
                  x_scale="unit", eta=0.05)
    W0, inp = I.initial_W(wl), I.step_inputs(wl, 1)
    W = to_dev(W0, torch)
    ctx = S.Context(config_for(wl, S.PREC_BF16), W)
    X, lab = to_dev(inp.X, torch), to_dev(inp.labels, torch)
    if per_worker:
        for p in reversed(range(workers)):
            r = slice(p * batch, (p + 1) * batch)
            ctx.sfb_compute_factors(p, X[r], None, lab[r])
        ctx.sfb_gather_factors()
        ctx.sfb_apply_update()
    else:
        ctx.sfb_step(X, None, lab)
    assert ctx.sfb_get_status() == 0
    assert torch.equal(ctx.operand_copy_as_tensor()[:, :cols], W.to(torch.bfloat16))
    Wg = W.cpu().numpy()
    ctx.close()
    err = rel_err(Wg, oracle_step(wl, W0, inp), W0)
    print(f"{rows} x {cols} K={wl.K}: rel err {err:.3e}")
    assert err <= TOL[S.PREC_BF16]


# One ragged tile, one row more than a tile, four full k-blocks and one pair more, several tiles per pair of CTAs.
@pytest.mark.parametrize("shape", [(5, 4, 1, 1), (257, 260, 4, 64), (257, 260, 1, 257), (1030, 2500, 5, 51), (6001, 2052, 2, 120)])
def test_update_forms(shape):
    check(*shape)


def plan(rows, cols, workers, batch, samples):
    return S.sfb_get_plan(S.make_config(S.MLR, rows, cols, workers, batch, 0.05, S.PREC_BF16), samples)


PAIRS = 2


# More than 128 samples, on pairs of CTAs or near the line between these and forward_kernel: long and short contractions, several rounds of
# tiles, the last sample and the last class alone in a tile.
@pytest.mark.parametrize("shape", [(873, 2800, 2, 317), (190, 708, 1, 513), (791, 9276, 4, 140), (9001, 4004, 2, 257), (10100, 5004, 5, 180),
                                   (2305, 1028, 1, 129)])
def test_logits_on_pairs(shape):
    check(*shape)


# (forward_kernel's size by now: of a shared-out tile the same is tested below.)
def test_logits_on_pairs_repeat():
    """The sums of a shared-out tile are in the order of the pairs: the same bits every time."""
    rows, cols, K = 9001, 4004, 514
    W0 = torch.randn(rows, cols, device="cuda") * 0.05
    X, lab = torch.randn(K, cols, device="cuda") / cols ** 0.5, torch.randint(0, rows, (K,), device="cuda", dtype=torch.int32)
    got = []
    for _ in range(2):
        W = W0.clone()
        ctx = S.Context(S.make_config(S.MLR, rows, cols, 1, K, 0.05, S.PREC_BF16), W)
        for _ in range(3):
            ctx.sfb_step(X, None, lab)
        assert ctx.sfb_get_status() == 0
        got.append(W)
        ctx.close()
    assert torch.equal(got[0], got[1])


# Those that are on pairs.  Whole tiles of 64 and 192 classes; a contraction shared out over most pairs, most of them in the middle of a
# tile; more tiles than pairs, the rest of the third round shared out; the last sample and the last class alone in a tile, whole
# and cut.
@pytest.mark.parametrize("shape", [(873, 2800, 2, 317), (65, 972, 1, 257), (791, 9276, 4, 140), (10100, 5004, 5, 180), (65, 1108, 1, 129),
                                   (257, 4188, 1, 129), (65, 4168, 1, 1025), (321, 4264, 1, 257)])
def test_logits_whose_plan_is_pairs(shape):
    assert plan(*shape, shape[2] * shape[3])[0] == PAIRS
    check(*shape)


# ... of samples behind the first ones: a worker's call, whose last tile overlaps the next worker's samples (whole tiles; cut ones, whose
# flags a call resets for the next).
@pytest.mark.parametrize("shape", [(873, 2800, 2, 317), (2220, 2588, 1, 144), (243, 4280, 2, 130), (257, 4332, 2, 129)])
def test_logits_on_pairs_of_workers(shape):
    assert plan(*shape, shape[3])[0] == PAIRS
    check(*shape, per_worker=True)


def test_logits_on_pairs_of_host_samples_in_parts():
    """512 samples of 4,000 features against 20,000 classes come in two parts of 256, whose tiles are cut: the loss and W of a step on the
    device, but for the rounding of sums in another order (operands in bf16: 2e-3 of the update)."""
    rows, cols, K = 20_000, 4_000, 512
    assert plan(rows, cols, 8, 64, 256) == (PAIRS, 2, 0)
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    W0 = torch.randn(rows, cols, generator=g, device="cuda") * 0.01
    X, lab = torch.randn(K, cols, generator=g, device="cuda") / cols ** 0.5, torch.randint(0, rows, (K,), generator=g, device="cuda", dtype=torch.int32)
    Xh, labh = X.cpu().pin_memory(), lab.cpu().pin_memory()
    got = []
    for host in (False, True):
        W = W0.clone()
        ctx = S.Context(S.make_config(S.MLR, rows, cols, 8, 64, 5.0, S.PREC_BF16), W)
        loss, status = ctx.sfb_step_host(Xh, None, labh) if host else (ctx.sfb_step(X, None, lab), 0)
        assert status == 0 and ctx.sfb_get_status() == 0
        got.append((W, loss if host else ctx.sfb_get_stats().last_loss))
        ctx.close()
    (Wd, ld), (Wh, lh) = got
    assert float((Wh - Wd).norm() / (Wd - W0).norm()) < 2e-3 and abs(lh - ld) < 1e-5 * ld


def test_logits_on_pairs_repeat_and_beside_another_context():
    """The sums of a shared-out tile are in the order of the pairs: the same bits every time, also where two contexts' kernels, each of
    which waits for pairs of its own, share the GPU."""
    rows, cols, K = 2500, 9000, 165
    assert plan(rows, cols, 1, K, K)[0] == PAIRS and plan(rows, cols, 1, K, K)[1] > 1
    W0 = torch.randn(rows, cols, device="cuda") * 0.05
    X, lab = torch.randn(K, cols, device="cuda") / cols ** 0.5, torch.randint(0, rows, (K,), device="cuda", dtype=torch.int32)
    torch.cuda.synchronize()

    def steps(contexts):
        streams = [torch.cuda.Stream() for _ in range(contexts)]
        Ws, ctxs = [W0.clone() for _ in streams], []
        torch.cuda.synchronize()
        for W, st in zip(Ws, streams):
            with torch.cuda.stream(st):
                ctxs.append(S.Context(S.make_config(S.MLR, rows, cols, 1, K, 0.05, S.PREC_BF16), W, stream=st))
        for _ in range(8):
            for ctx in ctxs:
                ctx.sfb_step(X, None, lab)
        for ctx in ctxs:
            assert ctx.sfb_get_status() == 0
            ctx.close()
        return Ws
    a, b, (c, d) = steps(1)[0], steps(1)[0], steps(2)
    assert torch.equal(a, b) and torch.equal(a, c) and torch.equal(a, d)


# Features that are no numbers or infinite stay with their samples: the factors of the others have the bits that they have without.
@pytest.mark.parametrize("shape", [(64, 256, 1, 40), (300, 3000, 1, 33), (873, 2800, 1, 317), (2500, 9000, 1, 165), (400, 260, 1, 100)])
@pytest.mark.parametrize("bad", [float("nan"), float("inf"), float("-inf")])
def test_features_that_are_not_finite(shape, bad):
    rows, cols, _, K = shape
    W0 = torch.randn(rows, cols, device="cuda") * 0.05
    X, lab = torch.randn(K, cols, device="cuda") / cols ** 0.5, torch.randint(0, rows, (K,), device="cuda", dtype=torch.int32)
    got = []
    for with_bad in (False, True):
        Xb = X.clone()
        if with_bad:
            Xb[K // 2, 5] = bad
        ctx = S.Context(S.make_config(S.MLR, rows, cols, 1, K, 0.05, S.PREC_BF16), W0.clone())
        ctx.sfb_step(Xb, None, lab)
        assert ctx.sfb_get_status() == 0
        got.append(ctx.factors_as_tensors()[0].clone())
        ctx.close()
    others = torch.arange(K, device="cuda") != K // 2
    assert torch.equal(got[0][others], got[1][others]) and bool(torch.isfinite(got[0]).all())
    mine = got[1][K // 2]
    assert bool(torch.isnan(mine[torch.arange(rows, device="cuda") != lab[K // 2]]).all())


# The logits of up to 64 samples: one sample, two classes; a contraction in 1, 2, 3 and 4 parts; the last tile of one class; 64 samples and 65;
# more classes than that, with few samples; samples of one call and of several workers.
@pytest.mark.parametrize("shape", [(2, 4, 1, 1), (200, 12004, 1, 37), (129, 68, 1, 33), (64, 256, 4, 32), (385, 1028, 3, 37), (4999, 3004, 2, 37), (7100, 516, 1, 17),
                                   (9000, 772, 2, 64), (9000, 772, 1, 65), (9473, 772, 1, 24), (15104, 132, 2, 9), (15105, 132, 2, 9)])
@pytest.mark.parametrize("per_worker", [False, True])
def test_logits_of_few_samples(shape, per_worker):
    check(*shape, per_worker=per_worker)


# The softmax of a small mini-batch in one launch: 128 samples and 129, one to eight partials and more, classes of one sample
# and (two classes) of more than eight; a class out of range; the update repeated on the sums that the launch keeps.
@pytest.mark.parametrize("shape", [(2, 1028, 1, 30), (64, 256, 4, 32), (250, 68, 1, 128), (250, 68, 1, 129), (1030, 260, 1, 40), (2000, 132, 1, 30)])
def test_merged_softmax(shape):
    check(*shape)


# Classes whose chain ends with a batch of eight samples, before it and behind it; followed ahead, and (with classes that have none) not.
@pytest.mark.parametrize("others", [0, 18])
def test_merged_softmax_chains(others):
    counts = [1, 7, 8, 9, 15, 16, 17, 30] + [0] * others
    rows, cols, K = len(counts), 1028, sum(counts)
    assert plan(rows, cols, 1, K, K)[2] == 1
    lab = torch.repeat_interleave(torch.arange(rows, device="cuda"), torch.tensor(counts, device="cuda"))[torch.randperm(K, device="cuda")].to(torch.int32)
    W0, X = torch.randn(rows, cols, device="cuda") * 0.03, torch.randn(K, cols, device="cuda") / 3
    W = W0.clone()
    ctx = S.Context(S.make_config(S.MLR, rows, cols, 1, K, 0.05, S.PREC_BF16), W)
    ctx.sfb_step(X, None, lab)
    assert ctx.sfb_get_status() == 0
    ctx.close()
    p = torch.softmax(X.double() @ W0.double().t(), 1)
    p[torch.arange(K, device="cuda"), lab.long()] -= 1
    step = -0.05 * p.t() @ X.double()
    err = ((W.double() - W0.double() - step).norm(dim=1) / step.norm(dim=1))[:8]     # operands in bf16: 2e-3 of a class's row
    assert float(err.max()) < 4e-3 and float((W.double() - W0.double() - step).norm() / step.norm()) < 2e-3


def test_merged_softmax_out_of_range_and_repeated():
    rows, cols, K = 40, 132, 50
    W0 = torch.randn(rows, cols, device="cuda") * 0.05
    X, lab = torch.randn(K, cols, device="cuda"), torch.randint(0, rows, (K,), device="cuda", dtype=torch.int32)
    lab[7], lab[8] = -1, rows
    got = []
    for repeats in (1, 2):
        W = W0.clone()
        ctx = S.Context(S.make_config(S.MLR, rows, cols, 1, K, 0.05, S.PREC_BF16), W)
        ctx.sfb_step(X, None, lab)
        for _ in range(repeats - 1):
            ctx.sfb_replay_update()
        assert ctx.sfb_get_status() == S.STATUS_LABEL_RANGE
        got.append(W.double())
        ctx.close()
    z = X.double() @ W0.double().t()
    p = torch.softmax(z, 1)
    ok = (lab >= 0) & (lab < rows)
    p[ok, lab[ok].long()] -= 1
    step = -0.05 * p.t() @ X.double()
    for n, W in enumerate(got, 1):                    # operands in bf16: 2e-3 of the update
        assert float((W - W0.double() - n * step).norm() / (n * step).norm()) < 2e-3


# Sparse samples staged and packed in one kernel (51,200 features, the most that it takes, and four more: in three), in one call and by workers:
# the bits of the dense samples' step.  Empty samples, a sample with an entry everywhere, one with a column out of range.
@pytest.mark.parametrize("cols", [4, 260, 51200, 51204])
@pytest.mark.parametrize("per_worker", [False, True])
def test_sparse_samples_as_dense_ones(cols, per_worker):
    rows, workers, batch = 70, 3, 5
    K = workers * batch
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    W0 = torch.randn(rows, cols, generator=g, device="cuda") * 0.05
    lab = torch.randint(0, rows, (K,), generator=g, device="cuda", dtype=torch.int32)
    got = []
    for sparse in (False, True):
        W = W0.clone()
        ctx = S.Context(S.make_config(S.MLR, rows, cols, workers, batch, 0.05, S.PREC_BF16, csr_nnz_max=K * cols + 1, csr_update=2), W)
        for t in range(2):                            # (another step's samples leave nothing behind)
            g.manual_seed(2 + t)
            X = torch.randn(K, cols, generator=g, device="cuda") * (torch.rand(K, cols, generator=g, device="cuda") < 0.05)
            X[3] = 0
            X[4] = 1
            parts = [slice(p * batch, (p + 1) * batch) for p in range(workers)] if per_worker else [slice(0, K)]
            for p, r in enumerate(parts):
                if sparse:
                    where = X[r].nonzero()
                    ptr = torch.zeros(X[r].shape[0] + 1, dtype=torch.int64, device="cuda")
                    ptr[1:] = torch.cumsum(torch.bincount(where[:, 0], minlength=X[r].shape[0]), 0)
                    idx, val = where[:, 1].to(torch.int32), X[r][where[:, 0], where[:, 1]]
                    if p == len(parts) - 1:           # one more entry of the last sample, out of range: skipped
                        ptr[-1] += 1
                        idx, val = torch.cat([idx, idx.new_tensor([cols])]), torch.cat([val, val.new_tensor([9.0])])
                    args = (ptr, idx.contiguous(), val.contiguous(), int(ptr[-1]), lab[r])
                    ctx.sfb_compute_factors_csr(p, *args) if per_worker else ctx.sfb_step_csr(*args)
                elif per_worker:
                    ctx.sfb_compute_factors(p, X[r], None, lab[r])
                else:
                    ctx.sfb_step(X, None, lab)
            if per_worker:
                ctx.sfb_gather_factors()
                ctx.sfb_apply_update()
        assert ctx.sfb_get_status() == (S.STATUS_INDEX_RANGE if sparse else 0)
        got.append(W)
        ctx.close()
    assert torch.equal(got[0], got[1])


# Sparse samples in more than one round of blocks, whose rows then have fewer threads: the bits of the dense samples' step.
@pytest.mark.parametrize("cols", [4, 252, 260, 4100])
def test_many_sparse_samples_as_dense_ones(cols):
    rows, K = 40, 700
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    W0 = torch.randn(rows, cols, generator=g, device="cuda") * 0.05
    lab = torch.randint(0, rows, (K,), generator=g, device="cuda", dtype=torch.int32)
    X = torch.randn(K, cols, generator=g, device="cuda") * (torch.rand(K, cols, generator=g, device="cuda") < 0.1)
    X[5] = 0
    X[6] = 1
    where = X.nonzero()
    ptr = torch.zeros(K + 1, dtype=torch.int64, device="cuda")
    ptr[1:] = torch.cumsum(torch.bincount(where[:, 0], minlength=K), 0)
    got = []
    for sparse in (False, True):
        W = W0.clone()
        ctx = S.Context(S.make_config(S.MLR, rows, cols, 1, K, 0.05, S.PREC_BF16, csr_nnz_max=K * cols, csr_update=2), W)
        if sparse:
            ctx.sfb_step_csr(ptr, where[:, 1].to(torch.int32).contiguous(), X[where[:, 0], where[:, 1]].contiguous(), int(ptr[-1]), lab)
        else:
            ctx.sfb_step(X, None, lab)
        assert ctx.sfb_get_status() == 0
        got.append(W)
        ctx.close()
    assert torch.equal(got[0], got[1])
