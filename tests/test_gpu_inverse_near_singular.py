"""Inverses of matrices close to singular, which the blocked elimination hands
to the step-by-step one: two rows of M equal up to a relative d, at sizes on
and off the panels' edges, beside a well-conditioned walker in the same call;
and an exactly singular one, which is refused."""
import numpy as np
import pytest

from paper_1711_11418_gb300 import inputs as I
from paper_1711_11418_gb300 import vmc

pytestmark = pytest.mark.gpu


def problem(N, d):
    p = I.make_problem("near", I.square(12, 12), 2 * N, sub=(1, 1), f_full=True, f_init="none",
                       noise=0.0)
    rng = np.random.default_rng(N)
    f = rng.standard_normal((p.Ns, p.Ns))
    f[1] = f[0] * (1.0 + d * rng.standard_normal(p.Ns))
    params = p.params.copy()
    params[p.n_g + p.n_v:] = f.reshape(-1)
    return p.copy_with(params=params), f, rng


def placement(rng, Ns, N, first):
    """Up electrons on the sites `first` and others from 2 on, down ones anywhere."""
    up = np.concatenate([first, 2 + rng.permutation(Ns - 2)[:N - len(first)]])
    return np.concatenate([up, rng.permutation(Ns)[:N]]).astype(np.int32)


@pytest.mark.parametrize("N", [25, 32, 81, 112, 127, 128])
@pytest.mark.parametrize("d", [1e-3, 1e-7])
@pytest.mark.parametrize("precision", [vmc.FP64, vmc.MIXED])
def test_inverse_close_to_singular(N, d, precision):
    p, f, rng = problem(N, d)
    cfg = np.array([placement(rng, p.Ns, N, [0]), placement(rng, p.Ns, N, [0, 1]),
                    placement(rng, p.Ns, N, [])], np.int32)
    with vmc.Context(p, 3, seed=5, precision=precision) as ctx:
        ctx.set_configs(cfg)
        got = [ctx.get_inverse(w) for w in range(3)]
    for w in range(3):
        M = f[np.ix_(cfg[w, :N], cfg[w, N:])]
        X, logdet, sign = got[w]
        ref = np.linalg.inv(M)
        # backward-stable elimination on both sides: |dX| <= const N eps cond |X|;
        # the mixed form's hi + lo words add 2^-46 of each entry
        tol = 64 * N * 2.3e-16 * np.linalg.cond(M) + (2.0 ** -46 if precision == vmc.MIXED else 0.0)
        assert np.linalg.norm(X - ref) <= tol * np.linalg.norm(ref)
        s, ld = np.linalg.slogdet(M)
        assert sign == int(s)
        assert abs(logdet - ld) <= 1e-10 * max(1.0, abs(ld)) + N * tol


def test_exactly_singular_is_refused():
    p, _, rng = problem(32, 0.0)
    with vmc.Context(p, 1, seed=5) as ctx:
        with pytest.raises(vmc.VmcError) as e:
            ctx.set_configs(np.array([placement(rng, p.Ns, 32, [0, 1])], np.int32))
            ctx.get_inverse(0)
        assert e.value.code == -4


@pytest.mark.parametrize("N", [25, 32, 33, 48])
@pytest.mark.parametrize("precision", [vmc.FP64, vmc.MIXED])
def test_small_inverses_by_panels(N, precision):
    """More walkers than SMs: N <= 48 goes by panels (fewer go step by step)."""
    p, f, rng = problem(N, 1e-3)
    W = 320
    cfg = np.array([placement(rng, p.Ns, N, []) for _ in range(W)], np.int32)
    with vmc.Context(p, W, seed=5, precision=precision) as ctx:
        ctx.set_configs(cfg)
        got = [ctx.get_inverse(w)[0] for w in range(0, W, 40)]
    for w, X in zip(range(0, W, 40), got):
        M = f[np.ix_(cfg[w, :N], cfg[w, N:])]
        ref = np.linalg.inv(M)
        tol = 64 * N * 2.3e-16 * np.linalg.cond(M) + (2.0 ** -46 if precision == vmc.MIXED else 0.0)
        assert np.linalg.norm(X - ref) <= tol * np.linalg.norm(ref)
