"""The Cholesky solve of an ill-conditioned S: backward error of the step no
larger than that of LAPACK's factorisation and substitution, at parameters whose
neighbours are nearly alike (the diagonal blocks themselves are ill-conditioned)
and at parameters that are nearly dependent across blocks."""
import numpy as np
import pytest
import scipy.linalg as sl

from paper_1711_11418_gb300 import inputs as I
from paper_1711_11418_gb300 import vmc

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53


def samples(kind, rows, Np, rng):
    if kind == "neighbours":   # correlation of parameters i, j: exp(-(i - j)^2 / 64)
        i = np.arange(Np)
        w, Q = np.linalg.eigh(np.exp(-((i[:, None] - i[None, :]) / 8.0) ** 2))
        return rng.standard_normal((rows, Np)) @ (Q * np.sqrt(w.clip(0))).T
    return rng.standard_normal((rows, 10)) @ rng.standard_normal((10, Np))


def backward_error(S, g, x):
    return np.linalg.norm(S @ x - g) / (np.linalg.norm(S, 2) * np.linalg.norm(x) + np.linalg.norm(g))


@pytest.mark.parametrize("kind", ["neighbours", "rank10"])
@pytest.mark.parametrize("shift", [1e-3, 1e-6, 1e-9, 1e-11])
@pytest.mark.parametrize("Np", [33, 64, 97, 300])
def test_cholesky_backward_error(kind, shift, Np):
    p = I.make_problem("sr", I.chain(8, 1), 4, U=4.0, sub=(2, 1), jastrow="none", noise=0.1, seed=1)
    p = p.copy_with(n_f=Np - 1, params=np.concatenate([p.params, np.ones(Np - 1 - p.n_f)]))
    rng = np.random.default_rng(Np)
    rows = 4 * Np
    O, E = samples(kind, rows, Np, rng), rng.standard_normal(rows)
    with vmc.Context(p, Np, seed=1, precision=vmc.FP64, max_samples=4) as ctx:
        ctx.set_samples(E, O)
        S, g = ctx.get_sr_matrices(shift, 0.0)
        ctx.set_params(np.zeros(Np))          # so that the new parameters are -x without rounding
        ctx.sr_step(1.0, shift, 0.0, solver=vmc.CHOLESKY)
        x = -ctx.get_params()
    L = np.linalg.cholesky(S)
    ref = sl.solve_triangular(L, sl.solve_triangular(L, g, lower=True), lower=True, trans=1)
    # the same method in another order of sums; S itself may differ in the last bits
    # between the two calls (atomic adds of its partial sums)
    assert backward_error(S, g, x) <= 16 * max(backward_error(S, g, ref), EPS)
