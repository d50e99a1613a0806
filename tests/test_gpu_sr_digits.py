"""The plain form's overlap matrix from 8-bit digit products, at the edges of
its tiles (64 parameters, 128 samples) and slabs, with columns of zeros, of one
value, and with entries far above the rest; and the Cholesky solve at the edges
of its 32-column panels."""
import numpy as np
import pytest

from paper_1711_11418_gb300 import inputs as I
from paper_1711_11418_gb300 import vmc

pytestmark = pytest.mark.gpu


def problem(n_f):
    """A chain whose layout has n_f pair parameters (1 Gutzwiller parameter beside)."""
    p = I.make_problem("sr", I.chain(8, 1), 4, U=4.0, sub=(2, 1), jastrow="none", noise=0.1, seed=1)
    extra = np.random.default_rng(0).uniform(-1, 1, n_f - p.n_f)
    return p.copy_with(n_f=n_f, params=np.concatenate([p.params, extra]))


def samples(rows, Np, seed):
    rng = np.random.default_rng(seed)
    O = rng.standard_normal((rows, Np)) * 2.0 ** rng.integers(-20, 21, (1, Np))
    O += 3.0 * np.abs(O).max(0, keepdims=True) * rng.standard_normal((1, Np))
    if Np > 20:
        O[:, 3] = 0.0
        O[:, 7] = -2.5
        O[rows // 2, 11] *= 1e4
    return rng.standard_normal(rows), O


@pytest.mark.parametrize("Np,rows", [(17, 1), (17, 3), (63, 15), (64, 127), (65, 128), (66, 129), (128, 255),
                                     (129, 1000), (200, 4099)])
def test_overlap_matrix(Np, rows):
    p = problem(Np - 1)
    E, O = samples(rows, Np, Np)
    with vmc.Context(p, -(-rows // 4), seed=1, precision=vmc.FP64, max_samples=4) as ctx:
        ctx.set_samples(E, O)
        S, _ = ctx.get_sr_matrices()
    X = O.astype(np.longdouble)
    X = X - X.mean(0)
    ref = (X.T @ X / rows).astype(np.float64)
    # entries of S against the columns' sizes; the centred samples are FP64
    # roundings of numbers of size |o| as well as of |O - o|
    size = np.sqrt(np.diag(ref)) + 2.3e-16 * np.abs(O).max(0) * 4
    assert np.all(np.abs(S - ref) <= 4e-14 * np.outer(size, size) + 8 * 2.3e-16 * (
        np.outer(np.abs(O).max(0) * 2.3e-16, np.abs(O).max(0)) + np.outer(np.sqrt(np.diag(ref)), np.abs(O).max(0))
        + np.outer(np.abs(O).max(0), np.sqrt(np.diag(ref)))))
    assert np.array_equal(S, S.T)


def test_overlap_matrix_in_slabs():
    """More samples than one slab of digits holds (1 GiB: 18432 at 4097 parameters)."""
    Np, rows = 4097, 18432 + 200
    p = problem(Np - 1)
    rng = np.random.default_rng(5)
    base = rng.standard_normal((rows, 64))
    O = np.empty((rows, Np))
    for k in range(0, Np, 64):
        O[:, k:k + 64] = np.roll(base, 17 * k, axis=0)[:, :min(64, Np - k)]
    with vmc.Context(p, rows // 4, seed=1, precision=vmc.FP64, max_samples=4) as ctx:
        ctx.set_samples(rng.standard_normal(rows), O)
        S, _ = ctx.get_sr_matrices()
    idx = np.concatenate([np.arange(0, 70), np.arange(2000, 2070), np.arange(4030, 4097)])
    X = O[:, idx] - O[:, idx].mean(0)
    ref = X.T @ X / rows
    assert np.abs(S[np.ix_(idx, idx)] - ref).max() <= 1e-13 * np.abs(np.diag(ref)).max()


@pytest.mark.parametrize("Np", [17, 31, 32, 33, 63, 64, 65, 96, 97, 300])
def test_cholesky_at_panel_edges(Np):
    rows = 3 * Np + 40
    p = problem(Np - 1)
    rng = np.random.default_rng(Np)
    O = rng.standard_normal((rows, Np)) * np.exp(rng.standard_normal((1, Np)))
    E = rng.standard_normal(rows) + O[:, :5].sum(1)
    with vmc.Context(p, -(-rows // 4), seed=1, precision=vmc.FP64, max_samples=4) as ctx:
        ctx.set_samples(E, O)
        S, g = ctx.get_sr_matrices(1e-3, 1e-4)
        p0 = ctx.get_params()
        ctx.sr_step(1.0, 1e-3, 1e-4, solver=vmc.CHOLESKY)
        x = p0 - ctx.get_params()
    ref = np.linalg.solve(S, g)
    # |dx| <= const n eps cond |x| for Cholesky; the step is read off parameters of order 1
    cond = np.linalg.cond(S)
    assert np.linalg.norm(x - ref) <= 16 * Np * 2.3e-16 * cond * np.linalg.norm(ref) + 1e-15 * np.sqrt(Np) * 4


def test_cholesky_reports_a_matrix_that_is_not_positive_definite():
    Np, rows = 70, 20          # rank deficient, no shift: a pivot is 0 up to rounding
    p = problem(Np - 1)
    rng = np.random.default_rng(1)
    O = np.zeros((rows, Np))
    O[:, :40] = rng.standard_normal((rows, 40))   # 30 columns of zeros: pivots exactly 0
    with vmc.Context(p, rows, seed=1, precision=vmc.FP64) as ctx:
        ctx.set_samples(rng.standard_normal(rows), O)
        p0 = ctx.get_params()
        with pytest.raises(vmc.VmcError) as e:
            ctx.sr_step(0.1, 0.0, 0.0, solver=vmc.CHOLESKY)
        assert e.value.code == -4
        assert np.array_equal(ctx.get_params(), p0)
