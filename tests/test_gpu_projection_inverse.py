"""From-scratch inverses of the projected state, FP64 form, where the matrix is
close to singular or of rows with entries of very different size: the
elimination by panels hands such a matrix to the step-by-step one, as for the
plain state.  The projection is onto the identity alone, so that the projected
ratio is the determinant's."""
import numpy as np
import pytest

from paper_1711_11418_gb300 import inputs as I
from paper_1711_11418_gb300 import vmc

pytestmark = pytest.mark.gpu

NS = 144


def context(f, cfg, N, seed=5):
    """A context with pair orbital f [NS, NS] on the placements cfg."""
    p = I.make_problem("near", I.square(12, 12), 2 * N, sub=(1, 1), f_full=True, f_init="none",
                       noise=0.0)
    rng = np.random.default_rng(seed)
    start = p.params.copy()
    start[p.n_g + p.n_v:] = rng.standard_normal(NS * NS)
    ctx = vmc.Context(p.copy_with(params=start), len(cfg), seed=seed, precision=vmc.FP64)
    ctx.set_projection(np.arange(NS, dtype=np.int32)[None, :], np.ones((1, NS), np.int8), np.ones(1))
    params = np.zeros(p.Np)
    params[p.n_g + p.n_v:] = f.reshape(-1)
    ctx.set_params(params)
    ctx.set_configs(np.array(cfg, np.int32))
    return ctx


@pytest.mark.parametrize("N", [25, 32, 81, 112, 128])
@pytest.mark.parametrize("d", [1e-3, 1e-7])
def test_projected_ratio_close_to_singular(N, d):
    rng = np.random.default_rng(N)
    f = rng.standard_normal((NS, NS))
    f[1] = f[0] * (1.0 + d * rng.standard_normal(NS))
    cfg = []
    for first in ([0], [0, 1]):
        up = np.concatenate([first, 2 + rng.permutation(NS - 2)[:N - len(first)]])
        cfg.append(np.concatenate([up, rng.permutation(NS)[:N]]))
    with context(f, cfg, N) as ctx:
        for w, c in enumerate(cfg):
            M = f[np.ix_(c[:N], c[N:])]
            X = np.linalg.inv(M)
            cond = np.linalg.cond(M)
            free = [t for t in range(NS) if t not in c[:N]][:4]
            moves = [(0, n, t) for n in (0, 1, N - 1) for t in free]
            got = ctx.eval_ratios(w, moves)
            ref = np.array([f[t, c[N:]] @ X[:, n] for _, n, t in moves])
            # backward-stable elimination: |dX| <= const N eps cond |X|, the sum adds N eps
            size = np.array([np.linalg.norm(f[t, c[N:]]) * np.linalg.norm(X, 2) for _, n, t in moves])
            assert np.all(np.abs(got - ref) <= 64 * N * 2.3e-16 * cond * size)


@pytest.mark.parametrize("N", [28, 40, 97])
def test_projected_rows_of_very_different_size(N):
    """Three rows of M with one panel's columns and one column behind it, the
    last row's second entry 2^-70 of its first: in fixed point under one exponent
    the second is lost and the column behind the panel has no pivot."""
    rng = np.random.default_rng(N)
    f = rng.standard_normal((NS, NS))
    e = 2.0 ** -70
    f[:3] = 0.0
    f[3:100, :3] = 0.0
    f[0, 0] = 1.0
    f[1, 1] = f[1, 2] = 1.0
    f[2, 0], f[2, 1] = 1.0, e
    up = np.concatenate([[0, 1, 2], 3 + rng.permutation(97)[:N - 3]])
    dn = 3 + rng.permutation(NS - 3)[:N]
    dn[0], dn[1], dn[20] = 0, 1, 2
    with context(f, [np.concatenate([up, dn])], N) as ctx:
        moves = [(0, 2, t) for t in range(100, 108)]
        got = ctx.eval_ratios(0, moves)
    # the inverse's column 2 is 1/e at the down electron on site 1, -1/e at the one on site 2
    ref = np.array([(f[t, 1] - f[t, 2]) / e for _, _, t in moves])
    assert np.all(np.abs(got - ref) <= 1e-12 * np.abs(ref) + 1e-10)
