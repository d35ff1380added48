"""The FP64 Gram block by exact products of digits on the tensor cores (rs_gram, RS_GRAM_F64, batches
large enough for that form) against extended precision, at the edges of its feature blocks (64) and
exact sums (256), with few and many versions, unaligned rows, and with elements that are no z-scores
(outside +-7.95, infinite, NaN), whose programs take plain FP64 multiply-adds.

Tolerance per entry: every element is rounded to 2^-52 (error 2^-53 each, so 2^-53 (sum |z_a| + sum
|z_b|)), the digit pairs left out are below 2^-54 per feature, and the sums of 256 features are rounded
and added in FP64 (two roundings of at most sum |z_a z_b| each)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


@pytest.fixture(scope="module")
def env():
    from paper_1910_07776_gb300 import build, rs
    build.build()
    ctx = rs.Context(0)
    yield rs, ctx
    ctx.close()


def _gram(rs, ctx, Z, P, V, F, gap=0):
    """K of P programs of V x F rows; `gap` elements between the programs' blocks."""
    dev = "cuda"
    ar = lambda n, s: torch.arange(n, device=dev, dtype=torch.int64) * s  # noqa: E731
    buf = torch.zeros(P, V * F + gap, dtype=torch.float64, device=dev)
    buf[:, :V * F] = torch.from_numpy(Z.reshape(P, V * F)).to(dev)
    b = rs.DeviceBatch(P, rs.RS_F64, P * V, V, F, buf.numel(), P * F, ar(P + 1, V),
                       torch.full((P,), F, dtype=torch.int32, device=dev), ar(P, V * F + gap), ar(P + 1, F),
                       buf.reshape(-1), torch.zeros(P * V, dtype=torch.uint8, device=dev),
                       torch.zeros(P * V, dtype=torch.float64, device=dev), None)
    K = torch.full((P * 64 * 64,), 7.0, dtype=torch.float64, device=dev)
    ctx.gram(b, rs.RS_GRAM_F64, K)
    torch.cuda.synchronize()
    ctx.check_device_status()
    return K.cpu().numpy().reshape(P, 64, 64)


def _check(K, Z, progs):
    V, F = Z.shape[1:]
    for p in progs:
        z = Z[p].astype(np.longdouble)
        ref, a = z @ z.T, np.abs(Z[p])
        row = a.sum(axis=1)
        bound = U * (row[:, None] + row[None]) + F * U / 2 + 2 * (F // 256 + 1) * U * (a @ a.T)
        assert np.all(np.abs(K[p, :V, :V] - ref) <= bound), p
        assert np.array_equal(K[p, :V, :V], K[p, :V, :V].T)
        assert np.all(K[p, V:] == 7.0) and np.all(K[p, :, V:] == 7.0)      # outside V x V: untouched


@pytest.mark.parametrize("V,F,P,gap", [(64, 1, 2600, 0), (64, 63, 60, 0), (64, 64, 60, 1), (33, 65, 150, 0), (5, 256, 400, 3),
                                       (64, 256, 20, 0), (64, 257, 20, 0), (40, 1030, 30, 1), (64, 4096, 12, 0)])
def test_entries_match_extended_precision(env, V, F, P, gap):
    rs, ctx = env
    rng = np.random.default_rng(V + F)
    Z = rng.standard_normal((P, V, F))
    Z = np.clip(Z, -7.9, 7.9)
    Z[0, 0] = 7.9                                            # the largest digits, all of one sign:
    Z[0, -1] = -7.9                                          # the longest exact sums
    Z[1] = np.where(rng.random((V, F)) < 0.5, 127.0 / 16, -127.0 / 16)
    Z[2] *= 2.0 ** rng.integers(-70, 1, size=(V, F))         # digits down to nothing
    Z[3] = 0.0
    Z[4] = np.tile(rng.standard_normal(F), (V, 1)).clip(-7.9, 7.9)
    _check(_gram(rs, ctx, Z, P, V, F, gap), Z, range(0, P, max(1, P // 12)) if P > 12 else range(P))
    _check(_gram(rs, ctx, Z[:5].repeat((P + 4) // 5, axis=0)[:P], P, V, F, gap),
           Z[:5].repeat((P + 4) // 5, axis=0)[:P], range(0, P, max(1, P // 10)))


def test_programs_of_other_values_take_plain_fp64(env):
    rs, ctx = env
    P, V, F = 40, 64, 130
    rng = np.random.default_rng(5)
    Z = rng.standard_normal((P, V, F)).clip(-6, 6)
    Z[3, 10, 129] = 9.5
    Z[7] *= 1e150
    Z[8, 63, 0] = np.inf
    Z[21, 0, 64] = np.nan
    Z[22, 5, 3] = -7.96
    K = _gram(rs, ctx, Z, P, V, F)
    _check(K, Z, [0, 2, 4, 6, 9, 20, 23, 39])
    for p in (3, 7, 8, 21, 22):                              # one FMA chain per entry, in feature order
        with np.errstate(all="ignore"):
            ref = Z[p].astype(np.longdouble) @ Z[p].astype(np.longdouble).T
        nan = np.isnan(ref)
        assert np.array_equal(np.isnan(K[p]), nan)
        fin = np.isfinite(ref)
        assert np.array_equal(np.isinf(K[p]), np.isinf(ref.astype(np.float64)) & ~nan)
        a = np.abs(np.where(np.isfinite(Z[p]), Z[p], 0))
        assert np.all(np.abs(K[p][fin] - ref[fin]) <= (F * U * (a @ a.T))[fin])


def test_programs_of_small_rows_keep_their_accuracy(env):
    """Digits hold an element to 2^-53 whatever its size, so a program with a row of norm below 1 (but not
    0) takes plain FP64 multiply-adds: the chain's bound, F roundings of at most sum |z_a z_b| (below the
    normal range of half the smallest subnormal), for it."""
    rs, ctx = env
    P, V, F = 40, 64, 130
    rng = np.random.default_rng(6)
    Z = rng.standard_normal((P, V, F)).clip(-6, 6)
    Z[3] *= 1e-8
    Z[5, 17] *= 1e-9                                         # one row of a program
    Z[7, 63] = 0.0                                           # a row of zeros: exact either way
    Z[9, 0] = rng.choice([-1.0, 1.0], F) * 2.0 ** -60        # digits of nothing
    Z[11] *= 1e-200
    Z[13, 40] /= 1.001 * np.linalg.norm(Z[13, 40])           # just below 1
    Z[15, 40] /= 0.999 * np.linalg.norm(Z[15, 40])           # just above: digits
    Z[17] = 0.0
    Z[19, 5] = 0.0
    Z[19, 5, 129] = 1e-3                                     # one element, the last
    K = _gram(rs, ctx, Z, P, V, F)
    _check(K, Z, [0, 2, 4, 6, 7, 8, 10, 12, 14, 15, 16, 17, 18, 20, 39])
    for p in (3, 5, 9, 11, 13, 19):
        z, a = Z[p].astype(np.longdouble), np.abs(Z[p])
        assert np.all(np.abs(K[p] - z @ z.T) <= F * (U * (a @ a.T) + 2.0 ** -1074)), p
        assert np.array_equal(K[p], K[p].T)


def test_ragged_programs(env):
    """1 to 64 versions and several widths in one batch, their z-scores."""
    from paper_1910_07776_gb300 import synth
    rs, ctx = env
    h = synth.make_batch(200, versions=(1, 64), feat_choices=[5, 64, 131, 300], dtype=np.float64, seed=8)
    b = rs.DeviceBatch.from_host(h)
    z = b.with_X(ctx.standardize(b))
    K = ctx.gram(z, rs.RS_GRAM_F64)
    torch.cuda.synchronize()
    ctx.check_device_status()
    K, Z = K.cpu().numpy().reshape(-1, 64, 64), z.X.cpu().numpy()
    for p in range(0, 200, 9):
        V, F, x0 = h.versions(p), int(h.feat_width[p]), int(h.x_offsets[p])
        a = Z[x0:x0 + V * F].reshape(V, F).astype(np.longdouble)
        row = np.abs(a).sum(axis=1)
        bound = U * (row[:, None] + row[None]) + F * U * (np.abs(a) @ np.abs(a).T + 0.5)
        assert np.all(np.abs(K[p, :V, :V] - a @ a.T) <= bound), p
