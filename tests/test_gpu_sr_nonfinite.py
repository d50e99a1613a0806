"""The plain form's overlap matrix where samples are infinite, not numbers, or
so large that products overflow: every entry is what FP64 arithmetic gives,
NaN, infinite or finite, and the columns beside are untouched."""
import warnings

import numpy as np
import pytest

from paper_1711_11418_gb300 import inputs as I
from paper_1711_11418_gb300 import vmc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Np,rows", [(17, 5), (65, 129), (200, 1000)])
def test_overlap_matrix_of_nonfinite_samples(Np, rows):
    p = I.make_problem("sr", I.chain(8, 1), 4, U=4.0, sub=(2, 1), jastrow="none", noise=0.1, seed=1)
    extra = np.random.default_rng(0).uniform(-1, 1, Np - 1 - p.n_f)
    p = p.copy_with(n_f=Np - 1, params=np.concatenate([p.params, extra]))
    rng = np.random.default_rng(Np)
    E, O = rng.standard_normal(rows), rng.standard_normal((rows, Np))
    clean = O.copy()
    O[rows // 2, 2] = np.nan
    O[:, 5] *= 1e-6
    O[rows - 1, 5] = np.nan            # beside small values
    O[0, 7] = np.inf
    O[0, 11] = -np.inf
    O[1 % rows, 11] = np.inf
    O[:, 13] *= 1e200                  # squares overflow, products with the others do not
    with vmc.Context(p, -(-rows // 4), seed=1, precision=vmc.FP64, max_samples=4) as ctx:
        ctx.set_samples(E, O)
        S, _ = ctx.get_sr_matrices()
        with pytest.raises(vmc.VmcError) as e:
            ctx.sr_step(0.1, 1e-3, 1e-4, solver=vmc.CHOLESKY)
        assert e.value.code == -4
        ctx.set_samples(E, clean)
        S2, _ = ctx.get_sr_matrices()
    with warnings.catch_warnings():
        warnings.simplefilter("ignore")
        X = O - O.mean(0)
        ref = np.einsum("ri,rj->ij", X, X) / rows
        X = clean - clean.mean(0)
    assert np.array_equal(np.isnan(S), np.isnan(ref))
    assert np.array_equal(np.isposinf(S), np.isposinf(ref)) and S[13, 13] == np.inf
    assert not np.isneginf(S).any()
    ok = np.isfinite(ref)
    size = np.linalg.norm(O[:, np.isfinite(O).all(0)] - O[:, np.isfinite(O).all(0)].mean(0), axis=0)
    full = np.zeros(Np)
    full[np.isfinite(O).all(0)] = size / np.sqrt(rows)
    with np.errstate(over="ignore"):
        tol = 4 * rows * 2.3e-16 * np.outer(full, full)
    assert np.all(np.abs(S[ok] - ref[ok]) <= tol[ok])
    # the next samples' matrix knows nothing of them
    ref2 = X.T @ X / rows
    d = np.sqrt(np.diag(ref2))
    assert np.all(np.abs(S2 - ref2) <= 4 * rows * 2.3e-16 * np.outer(d, d))
