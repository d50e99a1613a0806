"""The reciprocal of the eliminations by panels and of the Cholesky pivots:
diagonal matrices, whose inverse is the reciprocals themselves, within half a
unit in the last place of the exact ones."""
import numpy as np
import pytest

from paper_1711_11418_gb300 import inputs as I
from paper_1711_11418_gb300 import vmc

pytestmark = pytest.mark.gpu

NS, N = 144, 128


def relative_error(x, y):
    """|x y - 1| to first order, exactly enough: x y as two FP64 words."""
    def split(a):
        t = 134217729.0 * a
        h = t - (t - a)
        return h, a - h
    xh, xl = split(x)
    yh, yl = split(y)
    p = x * y
    e = ((xh * yh - p) + xh * yl + xl * yh) + xl * yl
    return np.abs((p - 1.0) + e)


@pytest.mark.parametrize("scale", [0, 1, -300, 300])
def test_reciprocals_of_a_diagonal_matrix(scale):
    p = I.make_problem("inv", I.square(12, 12), 2 * N, sub=(1, 1), f_full=True, f_init="none", noise=0.0)
    rng = np.random.default_rng(scale + 1000)
    start = p.params.copy()
    start[p.n_g + p.n_v:] = rng.standard_normal(NS * NS)
    W = 8
    cfg = []
    for _ in range(W):   # both electrons of a pair on one site: M is diagonal
        sites = rng.permutation(NS)[:N]
        cfg.append(np.concatenate([sites, sites]))
    with vmc.Context(p.copy_with(params=start), W, seed=5, precision=vmc.FP64) as ctx:
        for k in range(12):
            # sizes within 2^10 of each other: a larger spread goes to the step-by-step form
            d = rng.uniform(1.0, 2.0, NS) * 2.0 ** rng.integers(0, 10, NS) * rng.choice([-1.0, 1.0], NS)
            if k == 0:       # next to powers of two, and at them
                d[:6] = [1.0, 1.0 + 2.0 ** -52, 2.0 - 2.0 ** -52, 2.0, 4.0 / 3.0, 1.5]
            params = np.zeros(p.Np)
            params[p.n_g + p.n_v:] = np.diag(d * 2.0 ** scale).reshape(-1)
            ctx.set_params(params)
            ctx.set_configs(np.array(cfg, np.int32))
            for w in range(W):
                X, logdet, sign = ctx.get_inverse(w)
                x = d[cfg[w][:N]]
                y = np.diag(X) * 2.0 ** scale
                assert np.count_nonzero(X) == N
                assert relative_error(x, y).max() <= 2.0 ** -53 * (1.0 + 2.0 ** -20)
                assert sign == int(np.prod(np.sign(x)))
                want = np.log(np.abs(x)).sum() + N * scale * np.log(2.0)
                assert abs(logdet - want) <= 1e-12 * max(1.0, abs(want))
