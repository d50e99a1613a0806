"""The elimination by panels at small N, which only contexts of more walkers than
SMs take (fewer go step by step): rows and columns of very different size, and
matrices close to singular, handed over to the step-by-step form inside the same
launch, where both share the shared memory."""
import numpy as np
import pytest

from paper_1711_11418_gb300 import inputs as I
from paper_1711_11418_gb300 import vmc

pytestmark = pytest.mark.gpu

NS, W = 144, 320


def context(f, N, precision):
    p = I.make_problem("panels", I.square(12, 12), 2 * N, sub=(1, 1), f_full=True, f_init="none", noise=0.0)
    start = p.params.copy()
    start[p.n_g + p.n_v:] = np.random.default_rng(N).standard_normal(NS * NS)
    ctx = vmc.Context(p.copy_with(params=start), W, seed=5, precision=precision)
    params = np.zeros(p.Np)
    params[p.n_g + p.n_v:] = f.reshape(-1)
    ctx.set_params(params)
    return ctx


def placement(rng, N, first):
    up = np.concatenate([first, 2 + rng.permutation(NS - 2)[:N - len(first)]])
    return np.concatenate([up, rng.permutation(NS)[:N]]).astype(np.int32)


@pytest.mark.parametrize("N", [25, 31, 32, 33, 40, 47, 48, 49])
@pytest.mark.parametrize("d", [1e-3, 1e-7])
@pytest.mark.parametrize("precision", [vmc.FP64, vmc.MIXED])
def test_close_to_singular_among_ordinary_walkers(N, d, precision):
    rng = np.random.default_rng(N)
    f = rng.standard_normal((NS, NS))
    f[1] = f[0] * (1.0 + d * rng.standard_normal(NS))
    special = (3, 150, 151, 319)
    cfg = np.array([placement(rng, N, [0, 1] if w in special else []) for w in range(W)])
    look = special + (0, 2, 152, 318)
    with context(f, N, precision) as ctx:
        ctx.set_configs(cfg)
        got = {w: ctx.get_inverse(w) for w in look}
    for w in look:
        M = f[np.ix_(cfg[w, :N], cfg[w, N:])]
        X, logdet, sign = got[w]
        ref = np.linalg.inv(M)
        # backward-stable elimination on both sides; hi + lo words keep 2^-46
        tol = 64 * N * 2.3e-16 * np.linalg.cond(M) + (2.0 ** -46 if precision == vmc.MIXED else 0.0)
        assert np.linalg.norm(X - ref) <= tol * np.linalg.norm(ref)
        s, ld = np.linalg.slogdet(M)
        assert sign == int(s)
        assert abs(logdet - ld) <= 1e-10 * max(1.0, abs(ld)) + N * tol


@pytest.mark.parametrize("N", [25, 32, 33, 47, 48])
def test_graded_rows_and_columns(N):
    """Sizes apart by 2^24 in rows and in columns.  The inverse is compared after
    the sizes are divided out; partial pivoting does not know them, so the bound
    is that of numpy's elimination of the same graded matrix, which pivots alike."""
    rng = np.random.default_rng(7 * N)
    r, c = 2.0 ** rng.integers(-12, 13, NS), 2.0 ** rng.integers(-12, 13, NS)
    f = rng.standard_normal((NS, NS)) * r[:, None] * c[None, :]
    cfg = np.array([placement(rng, N, []) for _ in range(W)])
    look = list(range(0, W, 20))
    with context(f, N, vmc.FP64) as ctx:
        ctx.set_configs(cfg)
        got = {w: ctx.get_inverse(w)[0] for w in look}
    worst = numpy_worst = 0.0
    for w in look:
        up, dn = cfg[w, :N], cfg[w, N:]
        A = f[np.ix_(up, dn)] / r[up][:, None] / c[dn][None, :]
        ref = np.linalg.inv(A)
        err = lambda X: np.linalg.norm(X * r[up][None, :] * c[dn][:, None] - ref) / np.linalg.norm(ref) / np.linalg.cond(A)  # noqa: E731
        worst = max(worst, err(got[w]))
        numpy_worst = max(numpy_worst, err(np.linalg.inv(f[np.ix_(up, dn)])))
    assert worst <= 16 * max(numpy_worst, N * 2.3e-16)
