"""GPU parity of the Table 2 transfer (Sec. 5): rs_transfer through the C ABI against the FP64
CPU reference, for the six experiments on seeded stand-ins of the paper's runs, ragged runs,
both learners, float32 counters, RS_RANK_ALL and the degenerate fits.  IBK predictions,
rankings and counters are exact (a neighbour's label enters the mean unchanged, so only a
near-tie in distance could change a prediction).

Ridge: the two sides solve the same system by different FP64 algorithms (primal Cholesky on
the CPU, bordered dual LDL^T on the GPU), so they agree to about kappa * eps, kappa the
condition number of the fit.  The pooled z-scores of a group of N versions have trace(Z Z^T)
= N * F, so the largest eigenvalue of K + lambda I is at most N * F + lambda and
kappa <= 1 + N * F / lambda -- up to 1.8e7 for three runs of 64 versions and 96 features,
where the fixed 1e-9 relative bound of the other parity tests no longer holds.  Predictions
must agree within 1e-9 relative plus kappa_bound * eps * max(1, max |prediction|) absolute;
rankings equal outside decisions closer than four times that."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_1910_07776_gb300 import synth

from parity import close, compare_counters, compare_rankings

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rs():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1910_07776_gb300 import build
    build.build()
    from paper_1910_07776_gb300 import rs as _rs
    return _rs


@pytest.fixture(scope="module")
def ctx(rs):
    c = rs.Context(0)
    yield c
    c.close()


@pytest.fixture(scope="module")
def runs():
    return synth.make_runs(seed=0)


def _both(rs, ctx, train, test, groups, model, opt_mask=0x3F, flags=0, k=3, tau=1.05, lam=1e-3):
    f = flags | {"ibk": rs.RS_MODEL_IBK, "m5p": rs.RS_MODEL_M5P}.get(model, 0)
    g = rs.transfer_run(ctx, rs.DeviceBatch.from_host(train), rs.DeviceBatch.from_host(test), groups=groups,
                        lam=lam, k=k, tau=tau, flags=f, opt_mask=opt_mask)
    r = oracle.transfer(train, test, groups, lam=lam, k=k, tau=tau, flags=flags, opt_mask=opt_mask, model=model)
    g["abs_tol"] = _kappa_abs(train, test, groups, lam, r.pred_all)
    return g, r


def _kappa_abs(train, test, groups, lam, ref_pred):
    """The absolute tolerance of ridge predictions: kappa_bound * eps * prediction scale."""
    ro = train.row_offsets
    g = np.arange(test.n_programs + 1) if groups is None else np.asarray(groups)
    n_max = max(int(ro[g[q + 1]] - ro[g[q]]) for q in range(test.n_programs))
    kappa = 1.0 + n_max * int(train.feat_width.max()) / lam
    scale = max(1.0, float(np.nanmax(np.abs(ref_pred))) if np.isfinite(ref_pred).any() else 1.0)
    return max(1e-11, kappa * np.finfo(np.float64).eps * scale)


def _check(g, r, model, tau=1.05, abs_tol=1e-11):
    np.testing.assert_array_equal(g["fit_status"], r.fit_status)
    if model == "m5p":
        # the tree's discrete decisions (splits, dropped terms, pruning) come out the same; its
        # linear models are solved by another algorithm (Gauss-Jordan inverse and drop-one
        # updates against Cholesky refits), so the values agree to the node systems'
        # conditioning: 1e-7 relative
        close(g["pred_all"], r.pred_all, rel=1e-7, abs_=1e-9)
        nd, nn = compare_rankings(g["rec_code"], r.rec_code, r.pred_all, math.log(tau), tol=1e-6)
        compare_counters(g["counters"], r.counters, slack=nn)
        return
    if model == "ibk":
        np.testing.assert_array_equal(g["pred_all"], r.pred_all)
        np.testing.assert_array_equal(g["rec_code"], r.rec_code)
        np.testing.assert_array_equal(g["rec_pred"], r.rec_pred)
        np.testing.assert_array_equal(g["counters"], r.counters)
        return
    close(g["pred_all"], r.pred_all, abs_=abs_tol)
    nd, nn = compare_rankings(g["rec_code"], r.rec_code, r.pred_all, math.log(tau), tol=max(1e-8, 4 * abs_tol))
    compare_counters(g["counters"], r.counters, slack=nn)


@pytest.mark.parametrize("experiment", [1, 2, 3, 4, 5, 6])
@pytest.mark.parametrize("model", ["ridge", "ibk", "m5p"])
def test_table2_experiments(rs, ctx, runs, experiment, model):
    pr = synth.table2_problems(runs, experiment)
    g, r = _both(rs, ctx, pr.train, pr.test, pr.groups, model, opt_mask=pr.opt_mask)
    _check(g, r, model, abs_tol=g["abs_tol"])
    assert g["counters"][0] == pr.test.n_rows


@pytest.mark.parametrize("model", ["ridge", "ibk", "m5p"])
def test_ragged_runs_groups_float32_and_rank_all(rs, ctx, model):
    # groups of 1..4 ragged runs (1..64 versions, repeated widths), float32 counters, RANK_ALL
    b = synth.make_batch(40, versions=(1, 64), feat=33, dtype=np.float32, seed=77)
    rng = np.random.default_rng(77)
    sizes = rng.integers(1, 5, size=8)
    groups = np.concatenate([[0], np.cumsum(sizes)])
    train = synth.take_programs(b, list(range(int(groups[-1]))))
    test = synth.take_programs(b, list(range(30, 38)))
    for flags in (0, oracle.RANK_ALL):
        g, r = _both(rs, ctx, train, test, groups, model, opt_mask=0b011011, flags=flags, k=6, tau=0.9)
        _check(g, r, model, tau=0.9, abs_tol=g["abs_tol"])


@pytest.mark.parametrize("model", ["ridge", "ibk"])
def test_one_run_per_problem_default_groups(rs, ctx, runs, model):
    train = synth.take_programs(runs, [i for i, key in enumerate(runs.meta["index"]) if key[0] == "BH"][:12])
    test = synth.take_programs(runs, [i for i, key in enumerate(runs.meta["index"]) if key[0] == "BH"][6:18])
    g, r = _both(rs, ctx, train, test, None, model)
    _check(g, r, model, abs_tol=g["abs_tol"])


def test_degenerate_fits(rs, ctx):
    # a run of one version (every fit EMPTY) and a run of two versions one optimization apart
    # (one pair: the prediction is its label)
    X = np.exp(np.random.default_rng(0).normal(size=(3, 4)))
    mk = lambda rows, masks, lt: synth.ProgramBatch(
        X=X[rows].reshape(-1), x_offsets=np.array([0]), row_offsets=np.array([0, len(rows)]),
        feat_width=np.array([4], dtype=np.int32), masks=np.array(masks, dtype=np.uint8),
        log_time=np.array(lt), cycles=None)
    test = mk([0, 1, 2], [0, 1, 2], [0.0, -0.2, 0.1])
    for train in (mk([0], [0], [0.0]), mk([0, 1], [0, 1], [0.3, 0.1])):
        for model in ("ridge", "ibk", "m5p"):
            g, r = _both(rs, ctx, train, test, None, model)
            _check(g, r, model, abs_tol=g["abs_tol"])


def test_bad_group_is_reported_not_written(rs, ctx):
    # problem 1's group has a run of another feature width: RS_EDATA, its rows untouched,
    # problem 0 still computed
    b1 = synth.make_batch(3, versions=64, feat=16, seed=5)
    b2 = synth.make_batch(1, versions=64, feat=24, seed=6)
    train = synth.take_programs(b1, [0])
    both = synth.ProgramBatch(
        X=np.concatenate([train.X, b2.X]), x_offsets=np.array([0, train.X.size]), row_offsets=np.array([0, 64, 128]),
        feat_width=np.array([16, 24], dtype=np.int32), masks=np.concatenate([train.masks, b2.masks]),
        log_time=np.concatenate([train.log_time, b2.log_time]), cycles=np.concatenate([train.cycles, b2.cycles]))
    test = synth.take_programs(b1, [1, 2])
    dtr, dte = rs.DeviceBatch.from_host(both), rs.DeviceBatch.from_host(test)
    offs = torch.tensor([0, 1, 2], dtype=torch.int64, device="cuda")
    ws = ctx.workspace(ctx.transfer_workspace_bytes(dtr, dte, (offs, 1), rs.RS_MODEL_IBK))
    code = torch.full((128,), 0x7777, dtype=torch.int32, device="cuda")
    ctx.transfer(dtr, dte, ws, code, groups=(offs, 1), flags=rs.RS_MODEL_IBK)
    torch.cuda.synchronize()
    with pytest.raises(rs.RsError):
        ctx.check_device_status()
    c = code.cpu().numpy()
    assert (c[64:] == 0x7777).all() and (c[:64] != 0x7777).all()
    ref = oracle.transfer(train, synth.take_programs(b1, [1]), model="ibk")
    np.testing.assert_array_equal(c[:64].view(np.uint32), ref.rec_code)


@pytest.mark.parametrize("feat,runs_per,versions,case", [
    (1, 1, (3, 20), "plain"), (3, 2, (2, 64), "plain"), (17, 3, (10, 40), "ties"), (65, 1, (64, 64), "plain"),
    (100, 4, (60, 64), "plain"), (256, 2, (50, 64), "plain"), (40, 2, (30, 64), "equal"), (24, 3, (64, 64), "labels"),
    (70, 3, (64, 64), "many")])
def test_m5p_at_its_edges(rs, ctx, feat, runs_per, versions, case):
    """Trees of one to 128 instances, one to 256 attributes (more than a model takes terms), with equal
    attribute values and equal labels (ties between splits and between dropped terms are decided by
    the reference's own roundings), infinite labels, and labels that many attributes explain."""
    b = synth.make_batch(4 * runs_per + 4, versions=versions, feat=feat, dtype=np.float64, seed=500 + feat)
    rng = np.random.default_rng(feat)
    if case == "ties":            # counters of few distinct values; whole columns constant or repeated
        for p in range(b.n_programs):
            X = b.program_X(p)
            X[:] = np.exp(np.round(np.log(X / b.cycles[b.program_rows(p)][:, None])) * 0.5)
            X[:, 3] = X[:, 5]
            X[:, 7] = 2.0
        b.cycles = np.ones_like(b.cycles)
    if case == "equal":           # labels of two values only
        b.log_time = np.round(b.log_time)
    if case == "labels":
        b.log_time[int(b.row_offsets[1]) + 5] = np.inf
    if case == "many":            # every label a sum of many attributes' logs
        for p in range(b.n_programs):
            X = np.log(b.program_X(p) / b.cycles[b.program_rows(p)][:, None])
            b.log_time[b.program_rows(p)] = X @ rng.standard_normal(feat) / feat
    groups = np.arange(5, dtype=np.int64) * runs_per
    train = synth.take_programs(b, list(range(4 * runs_per)))
    test = synth.take_programs(b, list(range(4 * runs_per, 4 * runs_per + 4)))
    g, r = _both(rs, ctx, train, test, groups, "m5p", flags=oracle.RANK_ALL)
    _check(g, r, "m5p")


@pytest.mark.parametrize("gap", [1e-3, 1e-4, 1e-5, 1e-6])
@pytest.mark.parametrize("seed", [600, 601, 602])
def test_m5p_pairs_of_nearly_equal_counters(rs, ctx, gap, seed):
    """Counters in pairs that agree to `gap` of a deviation, on a few levels, so that a tree splits on both
    of a pair and its models drop one of them.  The versions predicted are training instances, where a
    model's values do not hang on the difference within a pair.  Tolerance: 100 kappa eps, kappa the
    condition of a pair's normal equations, at most 4 / gap^2 and, by the ridge of 1e-8, 2 x 96 / 1e-8 (the
    factor: the terms of a model and the deviations of the labels); a wrong drop moves predictions by up
    to tenths."""
    feat, runs_per = 16, 3
    b = synth.make_batch(4 * runs_per, versions=64, feat=feat, dtype=np.float64, seed=seed)
    rng = np.random.default_rng(seed)
    w = rng.standard_normal(feat // 2)
    for p in range(b.n_programs):
        level = np.round(1.5 * rng.standard_normal((64, feat // 2))) / 1.5
        b.program_X(p)[:] = np.exp(np.repeat(level, 2, axis=1) + gap * rng.standard_normal((64, feat)))
        b.log_time[b.program_rows(p)] = level @ w * 0.3 + 0.1 * rng.standard_normal(64)
    b.cycles = np.ones_like(b.cycles)
    test = synth.take_programs(b, [q * runs_per for q in range(4)])
    g, r = _both(rs, ctx, b, test, np.arange(5, dtype=np.int64) * runs_per, "m5p")
    tol = 100 * min(4 / gap ** 2, 2 * 96 / 1e-8) * np.finfo(np.float64).eps
    np.testing.assert_array_equal(g["fit_status"], r.fit_status)
    close(g["pred_all"], r.pred_all, rel=max(1e-7, tol), abs_=max(1e-9, tol))


def _m5p_on_its_rows(rs, ctx, train, test, groups):
    """rs_transfer's M5P predictions, and the reference's on the very rows that it standardized (they lie at
    the front of the workspace: the training rows, then from the next 256-byte boundary the test rows), so
    that only the trees are compared: {(problem, optimization): (got, reference, labels)}, all versions."""
    a, b = rs.DeviceBatch.from_host(train), rs.DeviceBatch.from_host(test)
    g = (torch.from_numpy(groups).cuda(), int(np.diff(groups).max()))
    flags = rs.RS_MODEL_M5P | rs.RS_RANK_ALL
    ws = ctx.workspace(ctx.transfer_workspace_bytes(a, b, g, flags))
    out = rs.alloc_outputs(test.n_rows, 0, 3)
    ctx.transfer(a, b, ws, out.rec_code, groups=g, flags=flags, pred_all=out.pred_all)
    torch.cuda.synchronize()
    ctx.check_device_status()
    raw, n = ws.view(torch.uint8), 8 * train.X.size
    ZA = raw[:n].view(torch.float64).cpu().numpy()
    ZB = raw[(n + 255) // 256 * 256:][:8 * test.X.size].view(torch.float64).cpu().numpy()
    pred, res = out.pred_all.cpu().numpy().reshape(-1, 6), {}
    rows = lambda Z, bt, p: Z[int(bt.x_offsets[p]):][:bt.versions(p) * bt.feat_width[p]].reshape(bt.versions(p), -1)  # noqa: E731
    for q in range(test.n_programs):
        for j in range(6):
            Zr, y = [], []
            for p in range(int(groups[q]), int(groups[q + 1])):
                m, lt = train.masks[train.program_rows(p)].astype(int), train.log_time[train.program_rows(p)]
                slot = {x: v for v, x in enumerate(m)}
                for v, x in enumerate(m):
                    if not (x >> j) & 1 and x | 1 << j in slot:
                        Zr.append(rows(ZA, train, p)[v])
                        y.append(lt[v] - lt[slot[x | 1 << j]])
            if y:
                ref = oracle.m5p_fit_predict(np.array(Zr), np.array(y), rows(ZB, test, q))[0]
                res[q, j] = pred[test.program_rows(q), j], ref, np.array(y)
    return res


@pytest.mark.parametrize("seed", [701, 703])
def test_m5p_counters_that_nearly_make_up_one_another(rs, ctx, seed):
    """Ten counters that are one of four others, or the sum of two, to 1e-6: every elimination starts from a
    nearly singular system.  Versions predicted and tolerance as in the test of pairs (the condition at most
    14 x 96 / 1e-8 by the ridge), and the trees are those of the same rows."""
    feat, runs_per, Q = 14, 3, 4
    b = synth.make_batch(Q * runs_per, versions=64, feat=feat, dtype=np.float64, seed=seed)
    rng = np.random.default_rng(seed)
    of, w = rng.integers(0, 4, size=(feat, 2)), rng.standard_normal(4)
    for p in range(b.n_programs):
        base = np.round(2 * rng.standard_normal((64, 4))) / 2
        x = np.empty((64, feat))
        x[:, :4] = base
        for f in range(4, feat):
            x[:, f] = x[:, of[f, 0]] + (x[:, of[f, 1]] if f % 2 else 0) + 1e-6 * rng.standard_normal(64)
        b.program_X(p)[:] = np.exp(x)
        b.log_time[b.program_rows(p)] = 0.3 * base @ w + 0.1 * rng.standard_normal(64)
    b.cycles = np.ones_like(b.cycles)
    test = synth.take_programs(b, [q * runs_per for q in range(Q)])
    tol = 100 * 14 * 96 / 1e-8 * np.finfo(np.float64).eps
    masks = test.masks.reshape(Q, 64).astype(int)
    for (q, j), (got, ref, _) in _m5p_on_its_rows(rs, ctx, b, test, np.arange(Q + 1, dtype=np.int64) * runs_per).items():
        trained = (masks[q] >> j) & 1 == 0
        close(got[trained], ref[trained], rel=1e-7, abs_=tol)


def test_m5p_splits_that_a_line_ties_with(rs, ctx):
    """Four instances, two on either value of the one counter: the split into halves and a line through
    their means have the same estimated error, (|y1 - y2| + |y3 - y4|) 3 / 4, whatever the labels, so that the
    roundings of both decide, and the tree follows the reference's.  The versions predicted lie between and
    beyond the two values, where a line and a split differ."""
    Q, masks = 200, np.arange(8, dtype=np.uint8)
    rng = np.random.default_rng(11)
    parity = (masks ^ masks >> 1 ^ masks >> 2) & 1           # 2 + 2 among the four before sides of each pair

    def batch(x):
        return synth.ProgramBatch(
            X=np.exp(x).reshape(-1), x_offsets=np.arange(Q, dtype=np.int64) * 8, row_offsets=np.arange(Q + 1, dtype=np.int64) * 8,
            feat_width=np.ones(Q, dtype=np.int32), masks=np.tile(masks, Q), log_time=rng.standard_normal(8 * Q), cycles=None)

    train = batch(rng.standard_normal((Q, 1)) + rng.standard_normal((Q, 1)) * parity)
    test = batch(rng.standard_normal((Q, 8)))
    res = _m5p_on_its_rows(rs, ctx, train, test, np.arange(Q + 1, dtype=np.int64))
    for q in range(Q):
        for j in range(3):
            got, ref, y = res[q, j]
            assert len(y) == 4
            close(got, ref, rel=1e-7, abs_=1e-7 * np.abs(ref).max())


@pytest.mark.parametrize("spread", [1e-2, 1e-4, 1e-5, 1e-6])
def test_m5p_labels_close_to_a_common_value(rs, ctx, spread):
    """Every optimization's speedup near one value: what the deviations of labels 1 +- spread are by the
    reference's arithmetic (sums of squares) is more and more its rounding, and its decisions are
    followed all the same."""
    runs_per = 3
    b = synth.make_batch(4 * runs_per + 4, versions=64, feat=24, dtype=np.float64, seed=610)
    bits = (np.arange(64)[:, None] >> np.arange(6)) & 1
    for p in range(b.n_programs):
        rows = b.program_rows(p)
        b.log_time[rows] = spread * b.log_time[rows] - bits[b.masks[rows]].sum(axis=1)
    train = synth.take_programs(b, list(range(4 * runs_per)))
    test = synth.take_programs(b, list(range(4 * runs_per, 4 * runs_per + 4)))
    g, r = _both(rs, ctx, train, test, np.arange(5, dtype=np.int64) * runs_per, "m5p", flags=oracle.RANK_ALL)
    _check(g, r, "m5p")


@pytest.mark.parametrize("feat,runs_per,versions,case", [
    (64, 1, (64, 64), "plain"), (72, 1, (2, 40), "plain"), (257, 1, (50, 64), "plain"), (33, 3, (64, 64), "plain"),
    (64, 2, (33, 64), "plain"), (129, 3, (1, 64), "plain"), (321, 4, (60, 64), "plain"), (96, 3, (64, 64), "far"),
    (96, 2, (40, 64), "nan")])
def test_ridge_blocks_at_the_edges_of_their_tiles(rs, ctx, feat, runs_per, versions, case):
    """Dot products by the tensor cores' blocks of 64 x 64 entries: part blocks, one and several stages of 64
    features and sums of 256, one to four runs; a test version far outside the training range (a counter
    e^40 times the others': its block takes plain FP64), and one whose counter is not a number."""
    Q = 6
    b = synth.make_batch(Q * runs_per + Q, versions=versions, feat=feat, dtype=np.float64, seed=900 + feat)
    train = synth.take_programs(b, list(range(Q * runs_per)))
    test = synth.take_programs(b, list(range(Q * runs_per, Q * runs_per + Q)))
    if case != "plain":
        for p in (1, 4):
            test.program_X(p)[-1, feat // 2] *= np.exp(40.0) if case == "far" else np.nan
    g, r = _both(rs, ctx, train, test, np.arange(Q + 1, dtype=np.int64) * runs_per, "ridge", flags=oracle.RANK_ALL)
    if case == "nan":             # that version's predictions alone are lost
        bad = [int(test.row_offsets[p + 1]) - 1 for p in (1, 4)]
        keep = np.setdiff1d(np.arange(test.row_offsets[-1]), bad)
        close(np.asarray(g["pred_all"]).reshape(-1, 6)[keep], np.asarray(r.pred_all).reshape(-1, 6)[keep], abs_=g["abs_tol"])
        return
    _check(g, r, "ridge", abs_tol=g["abs_tol"])


@pytest.mark.parametrize("feat", [40, 100, 300])
@pytest.mark.parametrize("case", ["one", "some", "all", "few_rows"])
def test_ridge_with_counters_outside_the_training_range(rs, ctx, feat, case):
    """Test versions whose counters lie far outside their training group's (z-scores beyond 15.9 enter the
    digit products as 0 and are added in FP64): one counter of every version, some, all, and single
    elements of a few versions; inside and outside values meet in one feature."""
    Q, runs_per = 5, 2
    b = synth.make_batch(Q * runs_per + Q, versions=(33, 64), feat=feat, dtype=np.float64, seed=950 + feat)
    rng = np.random.default_rng(feat)
    train = synth.take_programs(b, list(range(Q * runs_per)))
    test = synth.take_programs(b, list(range(Q * runs_per, Q * runs_per + Q)))
    for p in range(Q - 1):                       # (the last problem stays inside)
        X = test.program_X(p)
        if case == "few_rows":
            for v in (0, 7, X.shape[0] - 1):
                X[v, rng.integers(0, feat, size=3)] *= np.exp(rng.choice([-25.0, 30.0], size=3))
        else:
            cols = {"one": [feat - 1], "some": rng.choice(feat, feat // 3, replace=False), "all": np.arange(feat)}[case]
            X[:, cols] *= np.exp(rng.uniform(10.0, 30.0, size=len(cols)))
    g, r = _both(rs, ctx, train, test, np.arange(Q + 1, dtype=np.int64) * runs_per, "ridge", flags=oracle.RANK_ALL)
    _check(g, r, "ridge", abs_tol=g["abs_tol"])
