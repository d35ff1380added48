"""rs_standardize (A1) against its definition in extended precision: population z-scores of
log(max(x / c, 1e-30)) per program and feature, over block edges (1..64 versions, widths around
the 16- and 32-feature blocks), both element types, with and without cycle counts, extreme
exponents, and the values that leave the fixed-point logarithm's range (zeros, negatives,
subnormals, infinities, NaN).

Tolerance: each logarithm is within 0.625 units of 2^-53, the difference of two and the rounding
of the mean add to at most 2 units, and an element outside the fast range carries the two FP64
roundings of x (1 / c), 3 units; so a centred value is within 6 units of 2^-53, sigma within 6
units plus a relative 4 units, and z = d / sigma within (6 (1 + |z|) / sigma + 8 |z|) 2^-53."""
import numpy as np
import pytest
import torch

from paper_1910_07776_gb300 import synth

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


@pytest.fixture(scope="module")
def env():
    from paper_1910_07776_gb300 import build, rs
    build.build()
    ctx = rs.Context(0)
    yield rs, ctx
    ctx.close()


def _reference(x, c):
    with np.errstate(all="ignore"):
        q = x.astype(np.longdouble)
        if c is not None:      # FP64 range of the quotient: overflow is infinite
            q = q / c.astype(np.longdouble)[:, None]
            q = np.where(q > np.finfo(np.float64).max, np.longdouble(np.inf), q)
        l = np.log(np.where(q > np.longdouble(1e-30), q, np.longdouble(1e-30)))
        mu = l.mean(axis=0)
        sd = np.sqrt(((l - mu) ** 2).mean(axis=0))
        z = np.where(sd > 1e-12, (l - mu) / sd, 0)
    return z, mu, sd


def _batch(V, F, dtype, cyc, seed, wild, programs=3):
    rng = np.random.default_rng(seed)
    n = programs * V
    span = 30.0 if dtype == np.float32 or not wild else 650.0
    x = np.exp(rng.uniform(-span, span, size=(n, F)) if wild else rng.normal(20.0, 1.5, size=(n, F))).astype(dtype)
    if wild:
        bad = [0.0, -0.0, -3.5, np.nan, np.finfo(dtype).tiny / 4, np.finfo(dtype).max, np.finfo(dtype).tiny, 1e-30]
        for k, v in enumerate(bad):
            x[rng.integers(0, n), k % F] = dtype(v)
        x[rng.integers(0, V), F - 1] = dtype(np.inf)          # a feature of program 0 only
    x[V:2 * V, 0] = x[V, 0]                                   # a constant feature (raw counters)
    c = np.exp(rng.normal(15.0, 1.0, size=n)) if cyc else None
    if cyc:
        c[V:2 * V] = c[V]
        if wild:
            c[2 * V:] = np.exp(rng.uniform(-600, 600, size=n - 2 * V))
    masks = np.concatenate([np.sort(rng.choice(64, size=V, replace=False)) for _ in range(programs)])
    off = np.arange(programs + 1, dtype=np.int64) * V
    return synth.ProgramBatch(X=x.reshape(-1), x_offsets=off[:-1] * F, row_offsets=off,
                              feat_width=np.full(programs, F, dtype=np.int32), masks=masks.astype(np.uint8),
                              log_time=rng.normal(size=n), cycles=c)


@pytest.mark.parametrize("wild", [False, True])
@pytest.mark.parametrize("cyc", [False, True])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("V,F,programs", [(1, 1, 3), (2, 15, 3), (17, 16, 3), (33, 33, 3), (64, 40, 3), (64, 40, 160)])
def test_z_scores_match_the_definition(env, V, F, programs, dtype, cyc, wild):
    rs, ctx = env
    b = _batch(V, F, dtype, cyc, 7 * V + F, wild, programs)
    db = rs.DeviceBatch.from_host(b)
    mu = torch.empty(db.feat_total, dtype=torch.float64, device="cuda")
    sg = torch.empty_like(mu)
    Z = ctx.standardize(db, None, mu, sg).cpu().numpy().reshape(programs, V, F)
    ctx.check_device_status()
    mu, sg = mu.cpu().numpy().reshape(programs, F), sg.cpu().numpy().reshape(programs, F)
    for p in range(programs):
        z, m, s = _reference(b.program_X(p), None if b.cycles is None else b.cycles[b.program_rows(p)])
        inf = ~np.isfinite(m)
        assert np.array_equal(np.isinf(mu[p]), inf) and np.array_equal(np.isnan(sg[p]), inf)
        assert np.all(Z[p][:, inf] == 0)
        z, m, s = z[:, ~inf].astype(np.float64), m[~inf].astype(np.float64), s[~inf].astype(np.float64)
        assert np.all(np.abs(mu[p][~inf] - m) <= 6 * U * np.maximum(1, np.abs(m)))
        assert np.all(np.abs(sg[p][~inf] - s) <= 6 * U + 4 * U * s)
        const = s <= 1e-12
        assert np.all(Z[p][:, ~inf][:, const] == 0)
        live = s > 1e-9
        got, z, s = Z[p][:, ~inf][:, live], z[:, live], s[live]
        assert np.all(np.abs(got - z) <= (6 * (1 + np.abs(z)) / s + 8 * np.abs(z)) * U)
