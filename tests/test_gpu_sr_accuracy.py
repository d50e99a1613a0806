"""The plain form's overlap matrix to the accuracy that its digits keep: 56 bits
of every column, products to 2^-56 of the columns' largest entries, FP64 sums of
128 samples' exact ones."""
import numpy as np
import pytest

from paper_1711_11418_gb300 import inputs as I
from paper_1711_11418_gb300 import vmc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Np,rows", [(17, 127), (65, 129), (130, 1000), (200, 4099)])
@pytest.mark.parametrize("tails", [False, True])
def test_overlap_matrix_accuracy(Np, rows, tails):
    p = I.make_problem("sr", I.chain(8, 1), 4, U=4.0, sub=(2, 1), jastrow="none", noise=0.1, seed=1)
    p = p.copy_with(n_f=Np - 1, params=np.concatenate([p.params, np.ones(Np - 1 - p.n_f)]))
    rng = np.random.default_rng(Np + tails)
    O = rng.standard_normal((rows, Np)) * 2.0 ** rng.integers(-20, 21, (1, Np))
    if tails:
        O *= np.exp(rng.standard_normal((rows, Np)))
    E = rng.standard_normal(rows)
    with vmc.Context(p, -(-rows // 4), seed=1, precision=vmc.FP64, max_samples=4) as ctx:
        ctx.set_samples(E, O)
        S, _ = ctx.get_sr_matrices()
    X = O.astype(np.longdouble)
    X = X - X.mean(0)
    ref = np.einsum("ri,rj->ij", X, X) / rows
    d = np.sqrt(np.diag(ref))
    # rounding of the centred samples (2^-53 each, and of the mean) and of the FP64
    # sums: a few 2^-53 of sqrt(S_ii S_jj); heavy tails put more weight on one sample
    err = np.abs(S - ref) / np.outer(d, d)
    assert err.max() <= 2e-15
    assert np.sqrt((err ** 2).mean()) <= 2e-16
