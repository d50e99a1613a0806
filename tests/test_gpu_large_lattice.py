"""Inverses of few electrons on a large lattice, where the space per site is
larger than that of the elimination's staged operands: walkers fewer than the
SMs (step by step) and more (by panels), against numpy."""
import numpy as np
import pytest

from paper_1711_11418_gb300 import inputs as I
from paper_1711_11418_gb300 import vmc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [32, 48])
@pytest.mark.parametrize("W", [4, 200])
@pytest.mark.parametrize("precision", [vmc.FP64, vmc.MIXED])
def test_inverses_on_1024_sites(N, W, precision):
    p = I.make_problem("wide", I.square(32, 32), 2 * N, U=4.0, sub=(2, 2), jastrow="none", f_init="none",
                       noise=0.0)
    rng = np.random.default_rng(N)
    params = p.params.copy()
    params[p.n_g + p.n_v:] = rng.standard_normal(p.n_f)
    p = p.copy_with(params=params)
    f = p.f_matrix()
    with vmc.Context(p, W, seed=3, precision=precision) as ctx:
        ele, _ = ctx.get_configs()
        got = [ctx.get_inverse(w) for w in range(0, W, max(1, W // 8))]
        ctx.sample(1, 1, 1)
        after, _ = ctx.get_configs()
    for w, (X, logdet, sign) in zip(range(0, W, max(1, W // 8)), got):
        M = f[np.ix_(ele[w, :N], ele[w, N:])]
        ref = np.linalg.inv(M)
        # backward-stable elimination on both sides; hi + lo words keep 2^-46
        tol = 64 * N * 2.3e-16 * np.linalg.cond(M) + (2.0 ** -46 if precision == vmc.MIXED else 0.0)
        assert np.linalg.norm(X - ref) <= tol * np.linalg.norm(ref)
        s, ld = np.linalg.slogdet(M)
        assert sign == int(s)
        assert abs(logdet - ld) <= 1e-10 * max(1.0, abs(ld)) + N * tol
    for w in range(W):   # sites stay on the lattice, one electron of a spin each
        assert after[w].min() >= 0 and after[w].max() < p.Ns
        assert len(set(after[w, :N])) == N and len(set(after[w, N:])) == N
