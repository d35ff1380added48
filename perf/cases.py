"""Workloads of the recommendation tool's data-parallel path, as a user's program runs them: the
cross-validation step over every split of a batch of programs (ridge, closed-form
leave-one-version-out, IBK), the Table 2 transfer (ridge, IBK, M5P), pooled models over many
programs, and the learned surrogate (training and ranked inference).

Inputs follow the synthetic generator's recipe (``paper_1910_07776_gb300/synth.py``): latent
program states, main effects and pairwise interactions of six optimizations, log-normal counter
rates times cycle counts.  They are drawn on the GPU from the seed alone.
"""
import math
import zlib

import numpy as np
import torch

from paper_1910_07776_gb300 import rs

NOPT, LATENT, NMASK = 6, 8, 64
LAM, TAU, TOPK = 1e-3, 1.05, 3
DEV = "cuda"


# ------------------------------------------------------------------------------- the cases
def _cv(name, programs, vmin, vmax, feats, dtype, splits, nsplit, **more):
    d = dict(kind="cv", programs=programs, vmin=vmin, vmax=vmax, feats=feats, dtype=dtype, splits=splits,
             nsplit=nsplit, model="ridge", closed=False, precision="f64", rank_all=False, pack=False,
             pred_all=False, graph=False)
    d.update(more)
    return dict(d, name=name) if name else d


def listed():
    return [
        # one user's two programs, all 64 versions, the counters of one profiler run,
        # leave-one-version-out: the interactive call, where latency and launches count
        _cv("lovo_tiny", 2, 64, 64, "96", "f64", "lovo", 0, pred_all=True),
        # a handful of partly profiled programs with an odd counter set, Bernoulli splits, every
        # optimization ranked: odd, ragged sizes
        _cv("ragged_frac", 9, 3, 61, "131", "f64", "frac", 333, pred_all=True, rank_all=True),
        # the benchmark's batched cross-validation: 64 programs x 4096 half splits, one graph
        # launch per step
        _cv("half_batch", 64, 16, 64, "256", "f32", "half", 4096, graph=True),
        # the uneven stream: ten thousand programs of several counter widths, 1024 splits each
        _cv("uneven_stream", 10000, 8, 64, "64,128,256,512", "f32", "half", 1024, graph=True),
        # the paper's protocol (all masks, leave one version out) at the widest counter set
        _cv("lovo_wide", 256, 64, 64, "1024", "f64", "lovo", 0, pred_all=True),
        # the same protocol with the fits in closed form
        _cv("lovo_closed", 256, 64, 64, "1024", "f64", "lovo", 0, pred_all=True, closed=True),
        # the learner the paper chose, over the same protocol
        _cv("lovo_ibk", 256, 64, 64, "256", "f32", "lovo", 0, pred_all=True, model="ibk"),
        # Table 2, experiment 4 (six inputs, three runs each train; the other inputs are tested)
        dict(kind="transfer", model="ridge", inputs=6, runs=3, versions=64, feat=96, shared=False,
             name="transfer_ridge"),
        # the model tree on the measured n-body profile's shape (four inputs, three runs, 37 counters)
        dict(kind="transfer", model="m5p", inputs=4, runs=3, versions=64, feat=37, shared=False,
             name="transfer_m5p"),
        # one model per optimization over the pairs of 48 programs, ranking 16 held-out ones
        dict(kind="pooled", programs=48, held_out=16, vmin=16, vmax=64, feat=256, dtype="f32", name="pooled_fit"),
        # two epochs of the surrogate's training at its batch of 8192 rows
        dict(kind="train", rows=262144, batch=8192, steps=64, name="surrogate_train"),
        # ranked surrogate inference of a million versions with out-of-distribution flags
        dict(kind="infer", rows=1000000, chunk=131072, name="surrogate_infer"),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["lovo", "lovo", "lovo", "half", "half", "half", "transfer", "transfer", "pooled", "train", "infer"])
    if kind == "lovo":
        full = rng.random() < 0.5
        vmax = 64 if full else rng.randint(20, 64)
        way = rng.choice(["direct", "closed", "closed_bf16x3", "ibk"])
        return _cv(None, _logint(rng, 1, 256), 64 if full else rng.randint(4, vmax), vmax,
                   str(_logint(rng, 24, 1024)), rng.choice(["f32", "f64"]), "lovo", 0, pred_all=True,
                   closed=way.startswith("closed"), model="ibk" if way == "ibk" else "ridge",
                   precision="bf16x3" if way == "closed_bf16x3" else "f64")
    if kind == "half":
        programs = _logint(rng, 1, 3000)
        widths = [str(_logint(rng, 24, 512)) for _ in range(rng.choice([1, 1, 3]))]
        vmax = rng.randint(24, 64)
        graph = rng.random() < 0.5
        return _cv(None, programs, rng.randint(2, 24), vmax, ",".join(widths), rng.choice(["f32", "f64"]),
                   rng.choice(["half", "half", "frac"]), min(4096, _logint(rng, 1, max(2, 3000000 // programs))),
                   graph=graph, pack=rng.random() < 0.3, rank_all=rng.random() < 0.2,
                   model=rng.choice(["ridge", "ridge", "ridge", "ibk"]))
    if kind == "transfer":
        model = rng.choice(["ridge", "ibk", "m5p"])
        return dict(kind="transfer", model=model, inputs=rng.randint(2, 6), runs=rng.randint(1, 3),
                    versions=rng.randint(40, 64), feat=_logint(rng, 20, 64 if model == "m5p" else 160),
                    shared=rng.random() < 0.3)
    if kind == "pooled":
        return dict(kind="pooled", programs=_logint(rng, 12, 300), held_out=rng.randint(1, 40), vmin=rng.randint(16, 32),
                    vmax=rng.randint(40, 64), feat=_logint(rng, 33, 320), dtype=rng.choice(["f32", "f64"]))
    if kind == "train":
        batch = 8 * rng.randint(32, 1024)
        return dict(kind="train", rows=batch * rng.randint(1, 24) + rng.randint(0, 99), batch=batch,
                    steps=rng.randint(8, 64))
    return dict(kind="infer", rows=_logint(rng, 64, 1000000), chunk=rng.choice([8192, 32768, 131072]))


# ------------------------------------------------------------------------------- the inputs
_contexts = {}


def _ctx():
    """The process's one library handle, on torch's current stream, as a program keeps it."""
    if "ctx" not in _contexts:
        _contexts["ctx"] = rs.Context(0)
    return _contexts["ctx"]


def _gens(case, seed):
    """The case's own stream (which sizes a ragged batch has) and the seed's (every value)."""
    sizes = zlib.crc32(repr(sorted((k, v) for k, v in case.items() if k != "name")).encode())
    return np.random.Generator(np.random.PCG64(sizes)), torch.Generator(device=DEV).manual_seed(seed * 7919 + 13)


def _randn(g, *shape, dtype=torch.float64):
    return torch.randn(*shape, generator=g, device=DEV, dtype=dtype)


def _bits():
    m = torch.arange(NMASK, device=DEV)
    return ((m[:, None] >> torch.arange(NOPT, device=DEV)) & 1).double()


def _effects(g, h, w, u):
    """log speedups of the 64 masks of each program state h [P, 8], label noise included."""
    wn, un = w / w.norm(dim=1, keepdim=True), u / u.norm(dim=2, keepdim=True)
    a = 0.3 * h @ wn.T
    b = torch.triu(0.1 * torch.einsum("jkl,pl->pjk", un, h), diagonal=1)
    bits = _bits()
    return a @ bits.T + torch.einsum("vj,pjk,vk->pv", bits, b, bits) + 0.05 * _randn(g, h.shape[0], NMASK)


def _device_batch(X, V, F, masks, log_time, cycles):
    P = len(V)
    ro = np.concatenate([[0], np.cumsum(V)]).astype(np.int64)
    xo = np.concatenate([[0], np.cumsum(V * F)])[:-1].astype(np.int64)
    fo = np.concatenate([[0], np.cumsum(F)]).astype(np.int64)
    t = lambda a: torch.from_numpy(a).to(DEV)  # noqa: E731
    return rs.DeviceBatch(n_programs=P, dtype=rs.RS_F32 if X.dtype == torch.float32 else rs.RS_F64,
                          n_rows=int(ro[-1]), max_versions=int(V.max()), max_feat=int(F.max()),
                          x_elems=int(X.numel()), feat_total=int(fo[-1]), row_offsets=t(ro),
                          feat_width=t(F.astype(np.int32)), x_offsets=t(xo), feat_offsets=t(fo), X=X,
                          masks=masks.to(torch.uint8).contiguous(), log_time=log_time.contiguous(),
                          cycles=cycles.contiguous())


def _programs(P, vmin, vmax, feats, dtype, nrng, g):
    V = nrng.integers(vmin, vmax + 1, size=P).astype(np.int64)
    F = nrng.choice(np.asarray(feats, dtype=np.int64), size=P)
    fmax = int(F.max())
    w, u = _randn(g, NOPT, LATENT), _randn(g, NOPT, NOPT, LATENT)
    ft = torch.float32 if dtype == "f32" else torch.float64
    U, C = 0.5 * _randn(g, NOPT, fmax, dtype=ft), _randn(g, NOPT, fmax, LATENT, dtype=ft)
    M = math.sqrt(1.14 / LATENT) * _randn(g, fmax, LATENT, dtype=ft)
    h = _randn(g, P, LATENT)
    ls = _effects(g, h, w, u)
    lt = _randn(g, P, 1) - ls
    cyc = torch.exp(lt + 20.0 + 0.02 * _randn(g, P, NMASK))
    key = torch.rand(P, NMASK, generator=g, device=DEV)
    have = key.argsort(1).argsort(1) < torch.from_numpy(V).to(DEV)[:, None]
    masks = have.nonzero()[:, 1]
    xo = np.concatenate([[0], np.cumsum(V * F)])
    X = torch.empty(int(xo[-1]), dtype=ft, device=DEV)
    bits = _bits().to(ft)
    for f in np.unique(F):
        idx = np.nonzero(F == f)[0]
        step = max(1, int((1 << 27) // (NMASK * f)))
        for c in range(0, len(idx), step):
            ps = torch.from_numpy(idx[c:c + step]).to(DEV)
            hs = h[ps].to(ft)
            shift = U[None, :, :f] + 0.3 * torch.einsum("kfl,pl->pkf", C[:, :f], hs) / math.sqrt(LATENT)
            x = (hs @ M[:f].T)[:, None, :] + torch.matmul(bits[None], shift)
            x += 0.3 * _randn(g, len(ps), NMASK, int(f), dtype=ft)
            x = torch.exp(x) * cyc[ps][:, :, None].to(ft)
            hv = have[ps]
            start = torch.from_numpy(xo[idx[c:c + step]]).to(DEV)
            row = hv.cumsum(1) - 1
            at = (start[:, None] + row * int(f))[hv]
            X[(at[:, None] + torch.arange(int(f), device=DEV)).reshape(-1)] = x[hv].reshape(-1)
    return _device_batch(X, V, F, masks, lt[have], cyc[have])


def _splits(b, kind, n, nrng, g):
    V = (b.row_offsets[1:] - b.row_offsets[:-1])
    slots = torch.arange(NMASK, device=DEV)
    one = torch.ones((), dtype=torch.int64, device=DEV)
    weight = one << slots
    full = (weight[None] * (slots[None] < V[:, None])).sum(1)
    if kind == "lovo":
        vs = V.tolist()
        offs = torch.cat([torch.zeros(1, dtype=torch.int64, device=DEV), V.cumsum(0)])
        prog = torch.repeat_interleave(torch.arange(len(vs), device=DEV), V)
        slot = torch.arange(int(offs[-1]), device=DEV) - offs[prog]
        tm = full[prog] & ~(one << slot)
    else:
        offs = torch.arange(b.n_programs + 1, device=DEV) * n
        tm = torch.empty(b.n_programs * n, dtype=torch.int64, device=DEV)
        step = max(1, (1 << 20) // n)
        for p in range(0, b.n_programs, step):
            v = V[p:p + step]
            key = torch.rand(len(v), n, NMASK, generator=g, device=DEV)
            key = torch.where(slots < v[:, None, None], key, torch.full_like(key, 2.0))
            size = (v // 2)[:, None].expand(-1, n)
            if kind == "frac":      # every version with probability 1/2: how many, then which
                size = torch.from_numpy(nrng.binomial(v.cpu().numpy()[:, None], 0.5, size=(len(v), n))).to(DEV)
            sel = key.argsort(2).argsort(2) < size[..., None]
            tm[p * n:(p + len(v)) * n] = (sel * weight).sum(2).reshape(-1)
    pc = torch.zeros_like(tm)
    for k in range(NMASK):
        pc += (tm >> k) & 1
    per = torch.repeat_interleave(V, offs[1:] - offs[:-1])
    return rs.DeviceSplits(n_splits=int(tm.numel()), max_train=int(pc.max()), split_offsets=offs.contiguous(),
                           train_masks=tm.contiguous(), n_test_rows=int((per - pc).sum()))


def _runs(case, g):
    """The runs of each input of one code, as programs [inputs * runs] of the same versions."""
    I, R, V, F = case["inputs"], case["runs"], case["versions"], case["feat"]
    w, u = _randn(g, NOPT, LATENT), _randn(g, NOPT, NOPT, LATENT)
    U, C = 0.5 * _randn(g, NOPT, F), _randn(g, NOPT, F, LATENT)
    M = math.sqrt(1.14 / LATENT) * _randn(g, F, LATENT)
    h = _randn(g, 1, LATENT) + 0.4 * _randn(g, I, LATENT)
    scale = 0.6 + 0.4 * torch.arange(I, device=DEV)[:, None] / max(I - 1, 1)
    ls = scale * _effects(g, h, w, u)
    shift = U[None] + 0.3 * torch.einsum("kfl,pl->pkf", C, h) / math.sqrt(LATENT)
    x = (h @ M.T)[:, None, :] + torch.matmul(_bits()[None], shift) + 0.3 * _randn(g, I, NMASK, F)
    have = torch.rand(NMASK, generator=g, device=DEV).argsort().argsort() < V
    lt = (0.7 * torch.arange(I, device=DEV)[:, None, None] - ls[:, None]) + 0.01 * _randn(g, I, R, NMASK)
    cyc = torch.exp(lt + 20.0 + 0.02 * _randn(g, I, R, NMASK))
    X = torch.exp(x[:, None] + 0.05 * _randn(g, I, R, NMASK, F)) * cyc[..., None]
    masks = have.nonzero()[:, 0]
    return X[:, :, have].reshape(I * R, V, F), masks, lt[:, :, have].reshape(I * R, V), cyc[:, :, have].reshape(I * R, V)


def _take(runs, programs):
    X, masks, lt, cyc = runs
    P, V, F = len(programs), X.shape[1], X.shape[2]
    i = torch.tensor(programs, device=DEV)
    return _device_batch(X[i].reshape(-1).contiguous(), np.full(P, V, dtype=np.int64), np.full(P, F, dtype=np.int64),
                         masks.repeat(P), lt[i].reshape(-1), cyc[i].reshape(-1))


def _problems(case):
    """(runs that train, run that is tested): all runs of an input against every run of the others."""
    I, R = case["inputs"], case["runs"]
    return [([i * R + r for r in range(R)], i2 * R + r2) for i in range(I) for i2 in range(I) if i2 != i
            for r2 in range(R)]


def _mlp(g):
    dims, p = (256, 512, 512, 6), {}
    for i in range(3):
        s = 1.0 / math.sqrt(dims[i])
        p["W%d" % (i + 1)] = (2 * torch.rand(dims[i + 1], dims[i], generator=g, device=DEV) - 1) * s
        p["b%d" % (i + 1)] = (2 * torch.rand(dims[i + 1], generator=g, device=DEV) - 1) * s
    return p


def _rows(case, g):
    """Standardized rows and the labels of a smooth function of them."""
    n = case["rows"]
    X = _randn(g, n, 256)
    A = _randn(g, 256, NOPT, dtype=torch.float32) / 16.0
    Y = (0.4 * torch.tanh(X.float() @ A) + 0.05 * _randn(g, n, NOPT, dtype=torch.float32)).double()
    return X, Y


def _feats(case):
    return [int(f) for f in case["feats"].split(",")]


def _inputs(case, seed):
    nrng, g = _gens(case, seed)
    kind = case["kind"]
    if kind == "cv":
        b = _programs(case["programs"], case["vmin"], case["vmax"], _feats(case), case["dtype"], nrng, g)
        return b, _splits(b, case["splits"], case["nsplit"], nrng, g)
    if kind == "transfer":
        runs, probs = _runs(case, g), _problems(case)
        offs = torch.arange(len(probs) + 1, device=DEV) * case["runs"]
        return (_take(runs, [p for tr, _ in probs for p in tr]), _take(runs, [te for _, te in probs]),
                (offs.contiguous(), case["runs"]))
    if kind == "pooled":
        P = case["programs"]
        return (_programs(P, case["vmin"], case["vmax"], [case["feat"]], case["dtype"], nrng, g),
                _programs(case["held_out"], case["vmin"], case["vmax"], [case["feat"]], case["dtype"], nrng, g))
    X, Y = _rows(case, g)
    return X, Y, _mlp(g), torch.randint(0, NMASK, (case["rows"],), generator=g, device=DEV, dtype=torch.uint8)


def prepare(case, seed):
    ctx = _ctx()
    kind = case["kind"]
    st = {"case": case, "ctx": ctx}
    made = _inputs(case, seed)
    if kind == "cv":
        b, s = made
        R = s.n_test_rows
        st.update(b=b, s=s, ws=ctx.workspace(ctx.cv_workspace_bytes(b, s)),
                  out=rs.alloc_outputs(R, s.n_splits, TOPK, DEV, pred_all=case["pred_all"]))
        st["out"].rec_pred.zero_()
        st["flags"] = ((rs.RS_RANK_ALL if case["rank_all"] else 0) | (rs.RS_LOO_CLOSED if case["closed"] else 0) |
                       (rs.RS_MODEL_IBK if case["model"] == "ibk" else 0) | (rs.RS_PACK_PRED if case["pack"] else 0))
        st["precision"] = rs.RS_GRAM_BF16X3 if case["precision"] == "bf16x3" else rs.RS_GRAM_F64
        if case["graph"]:
            o = st["out"]
            st["graph"] = ctx.cv_graph(b, s, st["ws"], o.rec_offsets, o.rec_code, lam=LAM, k=TOPK, tau=TAU,
                                       flags=st["flags"], precision=st["precision"], rec_pred=o.rec_pred,
                                       pred_all=o.pred_all, counters=o.counters)
            o.counters.zero_()
    elif kind == "transfer":
        train, test, groups = made
        st.update(train=train, test=test, groups=groups, out=rs.alloc_outputs(test.n_rows, 0, TOPK, DEV))
        st["flags"] = {"ridge": 0, "ibk": rs.RS_MODEL_IBK, "m5p": rs.RS_MODEL_M5P}[case["model"]]
        st["fits"] = torch.empty(test.n_programs * NOPT, dtype=torch.uint8, device=DEV)
        st["ws"] = ctx.workspace(ctx.transfer_workspace_bytes(train, test, groups, st["flags"]))
    elif kind == "pooled":
        b, t = made
        st.update(b=b, t=t, ws=ctx.workspace(ctx.pooled_workspace_bytes(b)),
                  zb=b.with_X(torch.empty(b.x_elems, dtype=torch.float64, device=DEV)),
                  zt=t.with_X(torch.empty(t.x_elems, dtype=torch.float64, device=DEV)),
                  out=rs.alloc_outputs(t.n_rows, 0, TOPK, DEV))
    else:
        X, Y, par, masks = made
        sur = rs.Surrogate(ctx, case["batch"] if kind == "train" else 8192, infer_chunk=case.get("chunk", 0))
        sur.load({k: v.cpu().numpy() for k, v in par.items()})
        st.update(X=X, Y=Y, masks=masks, sur=sur)
        if kind == "train":
            st["loss"] = torch.zeros(case["steps"], device=DEV)
        else:
            n = case["rows"]
            if n >= 8192:      # the statistics of the rows that the surrogate was trained on
                sur.train(X, Y, steps=0)
            else:
                Xs = torch.cat([X, X.new_zeros(8192 - n, 256)])
                sur.train(Xs, Y.new_zeros(8192, NOPT), steps=0)
            st["code"] = torch.empty(n, dtype=torch.int32, device=DEV)
            st["rec_pred"] = torch.empty(n * TOPK, dtype=torch.float64, device=DEV)
    return st


# ------------------------------------------------------------------------------- one pass
def run(state):
    case, ctx = state["case"], state["ctx"]
    kind = case["kind"]
    if kind == "cv":
        o = state["out"]
        if "graph" in state:
            state["graph"].launch()
        else:
            ctx.cv_step(state["b"], state["s"], state["ws"], o.rec_offsets, o.rec_code, lam=LAM, k=TOPK, tau=TAU,
                        flags=state["flags"], precision=state["precision"], rec_pred=o.rec_pred, pred_all=o.pred_all,
                        counters=o.counters)
        res = {"rec_offsets": o.rec_offsets, "rec_code": o.rec_code, "rec_pred": o.rec_pred, "counters": o.counters}
        if o.pred_all is not None:
            res["pred_all"] = o.pred_all
        return res
    if kind == "transfer":
        o = state["out"]
        ctx.transfer(state["train"], state["test"], state["ws"], o.rec_code, groups=state["groups"], lam=LAM, k=TOPK,
                     tau=TAU, flags=state["flags"], opt_mask=0b110000 if case["shared"] else 0x3F,
                     fit_status=state["fits"], rec_pred=o.rec_pred, pred_all=o.pred_all, counters=o.counters)
        return {"rec_code": o.rec_code, "rec_pred": o.rec_pred, "pred_all": o.pred_all, "counters": o.counters,
                "fit_status": state["fits"]}
    if kind == "pooled":
        o = state["out"]
        ctx.standardize(state["b"], state["zb"].X)
        coef, fits = ctx.fit_pooled(state["zb"], None, lam=LAM, flags=rs.RS_REFINE_X, workspace=state["ws"])
        ctx.standardize(state["t"], state["zt"].X)
        ctx.predict_pooled(state["zt"], coef, fits, o.rec_code, k=TOPK, tau=TAU, rec_pred=o.rec_pred,
                           pred_all=o.pred_all, counters=o.counters)
        return {"coef": coef, "fit_status": fits, "rec_code": o.rec_code, "rec_pred": o.rec_pred,
                "pred_all": o.pred_all, "counters": o.counters}
    sur = state["sur"]
    if kind == "train":
        sur.train(state["X"], state["Y"], steps=case["steps"], lr=1e-3, weight_decay=0.01, use_graph=True,
                  loss_curve=state["loss"])
        res = {k: sur.view(k) for k in sur.NAMES}
        res.update({"grad_" + k: sur.view(k, "grad") for k in sur.NAMES})
        res["loss"] = state["loss"]
        return res
    pred, score, far = sur.infer(state["X"], ood_threshold=1.2, want_ood=True, masks=state["masks"], k=TOPK, tau=TAU,
                                 rec_code=state["code"], rec_pred=state["rec_pred"])
    return {"pred": pred, "score": score, "fallback": far, "rec_code": state["code"], "rec_pred": state["rec_pred"]}


# ------------------------------------------------------------------------------- the least work
def _pair_stats(V, train_frac):
    """Expected pairs per optimization of V random masks, and those with both versions trained on."""
    return 32.0 * V * (V - 1) / (NMASK * (NMASK - 1.0)) * train_frac


def work(case):
    kind = case["kind"]
    if kind == "cv":
        P, V = case["programs"], 0.5 * (case["vmin"] + case["vmax"])
        F = sum(_feats(case)) / len(_feats(case))
        es = 4 if case["dtype"] == "f32" else 8
        lovo = case["splits"] == "lovo"
        S = P * V if lovo else P * case["nsplit"]
        R = S if lovo else S * V / 2
        n = _pair_stats(V, (V - 2) / V if lovo else 0.25)
        cand = 6.0 if case["rank_all"] else 3.0
        byt = P * V * (F * es + 17) + S * 16 + R * (4 + 8 * TOPK + (48 if case["pred_all"] else 0))
        gram = P * V * V * F * (1.5 if case["model"] == "ibk" else 1.0)
        if case["model"] == "ibk":
            fits = R * cand * n
        elif case["closed"]:
            fits = P * NOPT * 2 * n ** 3 + R * cand * 8
        else:
            fits = S * NOPT * (n ** 3 / 3 + 3 * n * n) + R * cand * 2 * n
        return {"bytes": byt, "flops": gram + fits + P * V * F * 12}
    if kind == "transfer":
        I, R, V, F = case["inputs"], case["runs"], case["versions"], case["feat"]
        Q = I * (I - 1) * R
        n = R * _pair_stats(V, 1.0)
        nopt = 2 if case["shared"] else NOPT
        byt = Q * (R + 1) * V * F * 8 + Q * V * (4 + 8 * TOPK + 48)
        if case["model"] == "m5p":      # a sorted scan of every attribute at each level of the tree, and the node models
            fl = Q * nopt * (F * n * 12 * math.log2(max(n, 2)) + 4 * n * min(n, F) ** 2)
        else:
            fl = Q * (R * V) ** 2 * F * (0 if case["model"] == "ibk" else 1) + Q * V * R * V * F * 2
            fl += Q * nopt * (n ** 3 / 3) * (case["model"] == "ridge") + Q * V * 3 * 2 * n
        return {"bytes": byt, "flops": fl}
    if kind == "pooled":
        V, F = 0.5 * (case["vmin"] + case["vmax"]), case["feat"]
        es = 4 if case["dtype"] == "f32" else 8
        n = case["programs"] * _pair_stats(V, 1.0)
        rows = (case["programs"] + case["held_out"]) * V
        return {"bytes": rows * F * es + case["held_out"] * V * 76 + NOPT * (F + 1) * 8,
                "flops": NOPT * (n * F * F + F ** 3 / 3 + 8 * n * F) + case["held_out"] * V * 6 * F + rows * F * 12}
    par = 256 * 512 + 512 * 512 + 512 * 6
    if kind == "train":
        rows = case["batch"] * case["steps"]
        return {"bytes": rows * (256 + 6) * 8 + case["steps"] * par * 4 * 6, "flops": 6.0 * rows * par}
    return {"bytes": case["rows"] * (256 * 8 + 24 + 5 + 4 + 24 + 1) + par * 2, "flops": 2.0 * case["rows"] * par}


# ------------------------------------------------------------------------------- in 64 bits
def _padded(b):
    """Per program: standardized rows [P][64][F] by width, versions, masks, log times (padded)."""
    V = (b.row_offsets[1:] - b.row_offsets[:-1])
    P = b.n_programs
    slot = torch.arange(NMASK, device=DEV)
    on = slot[None] < V[:, None]
    row = b.row_offsets[:-1, None] + slot[None]
    row = torch.where(on, row, torch.zeros_like(row))
    masks = torch.where(on, b.masks[row].long(), torch.full_like(row, -1))
    return V, on, row, masks, torch.where(on, b.log_time[row], torch.zeros((), dtype=torch.float64, device=DEV))


def _z(x, c, on):
    """Population z-scores over the rows that are on of log(max(x / c, 1e-30))."""
    q = torch.log(torch.clamp(x / c[..., None], min=1e-30))
    n = on.sum(-1, keepdim=True)[..., None].double()
    q = q * on[..., None]
    mu = q.sum(-2, keepdim=True) / n
    d = (q - mu) * on[..., None]
    return d, mu, torch.sqrt((d * d).sum(-2, keepdim=True) / n)


def _blocks(b, dist):
    """The Gram block (or the block of squared distances) of every program, [P][64][64]."""
    V, on, row, masks, lt = _padded(b)
    K = torch.zeros(b.n_programs, NMASK, NMASK, dtype=torch.float64, device=DEV)
    for f in b.feat_width.unique().tolist():
        idx = (b.feat_width == f).nonzero()[:, 0]
        step = max(1, (1 << (20 if dist else 24)) // (NMASK * f))
        for ps in idx.split(step):
            at = b.x_offsets[ps, None] + torch.arange(NMASK, device=DEV)[None] * f
            at = torch.where(on[ps], at, torch.zeros_like(at))
            x = b.X[at[..., None] + torch.arange(f, device=DEV)].double()
            d, _, sd = _z(x, b.cycles[row[ps]], on[ps])
            z = torch.where(sd < 1e-12, torch.zeros_like(d), d / sd)
            K[ps] = torch.cdist(z, z, compute_mode="donot_use_mm_for_euclid_dist") ** 2 if dist else z @ z.mT
    return K, V, on, masks, lt


def _pairs(masks):
    """Pairs (v, v with j) of each program: before and after slots [P][6][32] and which exist."""
    P = masks.shape[0]
    slot_of = torch.full((P, NMASK + 1), -1, dtype=torch.long, device=DEV)
    slot_of.scatter_(1, torch.where(masks < 0, NMASK, masks), torch.arange(NMASK, device=DEV).expand(P, -1).contiguous())
    slot_of[:, NMASK] = -1
    before = torch.zeros(P, NOPT, 32, dtype=torch.long, device=DEV)
    after, have = torch.zeros_like(before), torch.zeros(P, NOPT, 32, dtype=torch.bool, device=DEV)
    for j in range(NOPT):
        lack = (masks >= 0) & ((masks >> j) & 1 == 0)
        w = torch.where(lack, slot_of.gather(1, torch.where(lack, masks | (1 << j), 0)), -1)
        ok = w >= 0
        order = torch.argsort((~ok).int(), dim=1, stable=True)[:, :32]
        before[:, j] = order
        after[:, j] = w.gather(1, order).clamp(min=0)
        have[:, j] = ok.gather(1, order)
    return before, after, have


def _ridge(M, m, y):
    """alpha and b of ridge with a free intercept, from M = K + lambda I; m [.., n] says which pairs train."""
    mm = m[..., :, None] * m[..., None, :]
    A = M * mm + torch.diag_embed(1.0 - m)
    L, _ = torch.linalg.cholesky_ex(A)
    s = torch.cholesky_solve(torch.stack([y * m, m], dim=-1), L)
    b = (m * s[..., 0]).sum(-1) / (m * s[..., 1]).sum(-1)
    return (s[..., 0] - b[..., None] * s[..., 1]) * m, b


def _nearest(d, m, y):
    """Mean label of the ten nearest of the pairs that train; d [.., rows, n]."""
    d = torch.where(m[..., None, :] > 0, d, torch.full_like(d, math.inf))
    k = min(10, d.shape[-1])
    near = torch.argsort(d, dim=-1, stable=True)[..., :k]
    lab = y[..., None, :].expand(d.shape).gather(-1, near)
    ok = torch.isfinite(d.gather(-1, near))
    return (lab * ok).sum(-1) / ok.sum(-1)


def _ranked(pred):
    """The reported lists of rows of predictions (NaN: no candidate), and how long each is."""
    p = torch.where(torch.isnan(pred) | (pred < math.log(TAU)), torch.full_like(pred, -math.inf), pred)
    top = torch.sort(p, dim=1, descending=True, stable=True)[0][:, :TOPK]
    return torch.where(torch.isinf(top), torch.full_like(top, math.nan), top), (~torch.isinf(top)).sum(1)


def _exact_cv(case, seed):
    b, s = _inputs(case, seed)
    if s.n_splits > 600000 or s.n_test_rows > 12000000:
        return None
    ibk = case["model"] == "ibk"
    if case["precision"] != "f64":
        return None      # the block itself is rounded to bfloat16 pieces: held to the start's outputs instead
    K, V, on, masks, lt = _blocks(b, ibk)
    before, after, have = _pairs(masks)
    P = b.n_programs
    pi = torch.arange(P, device=DEV)[:, None, None]
    y = lt[pi, before] - lt[pi, after]
    prog = torch.repeat_interleave(torch.arange(P, device=DEV), s.split_offsets[1:] - s.split_offsets[:-1])
    out = []
    for at in torch.arange(s.n_splits, device=DEV).split(8192):
        p, tm = prog[at], s.train_masks[at]
        train = ((tm[:, None] >> torch.arange(NMASK, device=DEV)) & 1).bool() & on[p]
        pred = torch.full((len(at), NMASK, NOPT), math.nan, dtype=torch.float64, device=DEV)
        ci = torch.arange(len(at), device=DEV)[:, None]
        for j in range(NOPT):
            bf, af = before[p, j], after[p, j]
            m = (have[p, j] & train[ci, bf] & train[ci, af]).double()
            Kx = K[p].gather(2, bf[:, None, :].expand(-1, NMASK, -1))
            if ibk:
                v = _nearest(Kx, m, y[p, j])
            else:
                M = Kx.gather(1, bf[:, :, None].expand(-1, -1, 32)) + LAM * torch.eye(32, dtype=torch.float64, device=DEV)
                alpha, b0 = _ridge(M, m, y[p, j])
                v = b0[:, None] + (Kx * alpha[:, None, :]).sum(2)
            ok = (m.sum(1) > 0)[:, None]
            if not case["rank_all"]:
                ok = ok & ((masks[p] >> j) & 1 == 0)
            pred[:, :, j] = torch.where(ok, v, math.nan)
        out.append(pred[on[p] & ~train])
    pred = torch.cat(out)
    rec, n = _ranked(pred)
    if case["pack"]:
        flat = torch.zeros(rec.numel(), dtype=torch.float64, device=DEV)
        got = rec[~torch.isnan(rec)]
        flat[:got.numel()] = got
        rec = flat
    res = {"rec_offsets": None, "rec_code": None, "rec_pred": rec.reshape(-1), "counters": None}
    if case["pred_all"]:
        res["pred_all"] = pred.reshape(-1)
    return res


def _exact_transfer(case, seed):
    if case["model"] == "m5p":
        return None
    train, test, _ = _inputs(case, seed)
    R, V, F, Q = case["runs"], case["versions"], case["feat"], test.n_programs
    x = train.X.double().reshape(Q, R * V, F)
    on = torch.ones(Q, R * V, dtype=torch.bool, device=DEV)
    d, mu, sd = _z(x, train.cycles.reshape(Q, R * V), on)
    zt = torch.log(torch.clamp(test.X.double().reshape(Q, V, F) / test.cycles.reshape(Q, V, 1), min=1e-30)) - mu
    z, zt = (torch.where(sd < 1e-12, torch.zeros_like(t), t / sd) for t in (d, zt))
    masks = test.masks[:V].long()
    before, after, have = _pairs(torch.cat([masks, torch.full((NMASK - V,), -1, device=DEV)])[None])
    lt = train.log_time.reshape(Q, R, V)
    pred = torch.full((Q, V, NOPT), math.nan, dtype=torch.float64, device=DEV)
    for j in range(NOPT):
        if case["shared"] and not (0b110000 >> j) & 1:
            continue
        bf, af = before[0, j][have[0, j]], after[0, j][have[0, j]]
        if not len(bf):
            continue
        rows = (torch.arange(R, device=DEV)[:, None] * V + bf[None]).reshape(-1)
        y = (lt[:, :, bf] - lt[:, :, af]).reshape(Q, -1)
        zp, m = z[:, rows], torch.ones(Q, len(rows), dtype=torch.float64, device=DEV)
        if case["model"] == "ibk":
            v = _nearest(torch.cdist(zt, zp, compute_mode="donot_use_mm_for_euclid_dist") ** 2, m, y)
        else:
            alpha, b0 = _ridge(zp @ zp.mT + LAM * torch.eye(len(rows), dtype=torch.float64, device=DEV), m, y)
            v = b0[:, None] + (zt @ (zp.mT @ alpha[..., None]))[..., 0]
        pred[:, :, j] = torch.where((masks >> j) & 1 == 0, v, math.nan)
    pred = pred.reshape(-1, NOPT)
    return {"rec_code": None, "rec_pred": _ranked(pred)[0].reshape(-1), "pred_all": pred.reshape(-1), "counters": None,
            "fit_status": None}


def _exact_pooled(case, seed):
    b, t = _inputs(case, seed)
    f = case["feat"]

    def rows(batch):
        V, on, row, masks, lt = _padded(batch)
        x = batch.X.double().reshape(-1, f)[row]
        d, _, sd = _z(x, batch.cycles[row], on)
        return torch.where(sd < 1e-12, torch.zeros_like(d), d / sd), on, masks, lt

    z, on, masks, lt = rows(b)
    zt, ont, maskt, _ = rows(t)
    before, after, have = _pairs(masks)
    coef = torch.empty(NOPT, f + 1, dtype=torch.float64, device=DEV)
    pi = torch.arange(b.n_programs, device=DEV)[:, None].expand(-1, 32)
    for j in range(NOPT):
        ok = have[:, j]
        c = z[pi[ok], before[:, j][ok]]
        y = lt[pi[ok], before[:, j][ok]] - lt[pi[ok], after[:, j][ok]]
        cm, ym = c.mean(0), y.mean()
        G = (c - cm).T @ (c - cm) + LAM * torch.eye(f, dtype=torch.float64, device=DEV)
        L = torch.linalg.cholesky(G)
        beta = torch.cholesky_solve(((c - cm).T @ (y - ym))[:, None], L)[:, 0]
        coef[j, 0], coef[j, 1:] = ym - cm @ beta, beta
    pred = zt[ont] @ coef[:, 1:].T + coef[:, 0]
    pred = torch.where((maskt[ont][:, None] >> torch.arange(NOPT, device=DEV)) & 1 == 0, pred, math.nan)
    return {"coef": coef, "fit_status": None, "rec_code": None, "rec_pred": _ranked(pred)[0].reshape(-1),
            "pred_all": pred.reshape(-1), "counters": None}


def _forward(p, x):
    h = torch.nn.functional.gelu(x @ p["W1"].T + p["b1"], approximate="tanh")
    h = torch.nn.functional.gelu(h @ p["W2"].T + p["b2"], approximate="tanh")
    return h @ p["W3"].T + p["b3"]


def _exact_train(case, seed):
    X, Y, par, _ = _inputs(case, seed)
    p = {k: v.double().requires_grad_(True) for k, v in par.items()}
    opt = torch.optim.AdamW(list(p.values()), lr=1e-3, betas=(0.9, 0.999), eps=1e-8, weight_decay=0.01)
    per, loss = case["rows"] // case["batch"], []
    n, at = case["batch"], 0
    if case["rows"] % n:
        return None      # where the minibatches wrap around is the library's own affair
    for i in range(case["steps"]):
        at = (i % per) * n
        opt.zero_grad()
        e = ((_forward(p, X[at:at + n]) - Y[at:at + n]) ** 2).mean()
        e.backward()
        opt.step()
        loss.append(e.detach())
    res = {k: v.detach() for k, v in p.items()}
    for k in ("W3", "b3"):
        full = torch.zeros(16, *res[k].shape[1:], dtype=torch.float64, device=DEV)
        full[:NOPT] = res[k]
        res[k] = full
    res.update({"grad_" + k: None for k in p})      # what is left of a gradient after the steps is rounding's own
    res["loss"] = torch.stack(loss)
    return res


def _exact_infer(case, seed):
    X, Y, par, masks = _inputs(case, seed)
    p = {k: v.double() for k, v in par.items()}
    pred = torch.cat([_forward(p, x) for x in X.split(65536)])
    n = case["rows"]
    stat = X if n >= 8192 else torch.cat([X, X.new_zeros(8192 - n, 256)])
    mu, sd = stat.mean(0), stat.std(0, unbiased=False)
    score = torch.cat([(((x - mu) / sd) ** 2).mean(1) for x in X.split(65536)])
    return {"pred": pred, "score": score, "fallback": None, "rec_code": None, "rec_pred": None}


def exact(case, seed):
    return {"cv": _exact_cv, "transfer": _exact_transfer, "pooled": _exact_pooled, "train": _exact_train,
            "infer": _exact_infer}[case["kind"]](case, seed)
