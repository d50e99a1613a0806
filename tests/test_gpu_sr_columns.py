"""Column sums of the samples (means, force, diagonal of S) at row counts around
the reduction's chunks and unrolling, with zeros and subnormal entries
among the samples, against numpy.

Force: a sum of `rows` products in FP64 of the stored samples.  Diagonal: through
one conjugate-gradient step with a large relative shift, x = g (g.g) / (g.S~ g)."""
import numpy as np
import pytest

from paper_1711_11418_gb300 import inputs as I
from paper_1711_11418_gb300 import vmc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [2, 3, 17, 63, 65, 255, 257, 1027])
@pytest.mark.parametrize("precision", [vmc.FP64, vmc.MIXED])
def test_force_and_diagonal_by_rows(rows, precision):
    p = I.make_problem("cols", I.chain(18, 1), 10, U=4.0, f_full=True, jastrow="chain", noise=0.3,
                       seed=3)
    rng = np.random.default_rng(rows)
    Np = p.Np
    O = rng.standard_normal((rows, Np)) * 2.0 ** rng.integers(-6, 7, Np)
    O[:, 1::5] *= rng.random((rows, len(range(1, Np, 5)))) < 0.5     # zeros of both signs
    O[0, 1::5] = -0.0
    O[:, 2] = 1e-41 * np.arange(1, rows + 1)                         # subnormal in FP32
    O[:, 3] *= 50.0
    E = rng.standard_normal(rows) - 7.0
    if precision == vmc.MIXED:
        O = O.astype(np.float32).astype(np.float64)
    with vmc.Context(p, rows, seed=1, precision=precision, max_samples=1) as ctx:
        ctx.set_samples(E, O)
        _, g = ctx.get_sr_matrices(with_S=False)
        before = ctx.get_params()
        rel, absolute, dtau = 50.0, 1e-3, 1.0
        ctx.sr_step(dtau, rel, absolute, solver=vmc.CG, cg_eps=1e-30, cg_kmax=1)
        x = (before - ctx.get_params()) / dtau
    Z, e = O - O.mean(0), E - E.mean()
    want = Z.T @ e / rows
    # FP64 sums in another order, and a mean off by rows eps
    tol = 4 * rows * 2.3e-16 * (np.abs(Z) + np.abs(O.mean(0))).T @ (np.abs(e) + np.abs(E.mean())) / rows
    assert np.all(np.abs(g - want) <= tol + 1e-300)
    Sg = Z.T @ (Z @ g) / rows + rel * (Z * Z).mean(0) * g + absolute * g
    step = g * (g @ g) / (g @ Sg)
    # the mixed form's FP32 products of 16 terms add 2^-20 of the part without the shift
    tol = 1e-10 if precision == vmc.FP64 else 1e-5
    assert np.linalg.norm(x - step) <= tol * np.linalg.norm(step) + 2.3e-16 * np.linalg.norm(before)
