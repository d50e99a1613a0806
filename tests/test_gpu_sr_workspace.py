"""The workspace of the plain form's overlap matrix in a batch: one per solver
stream, whatever the number of systems, with systems of different sizes taking
turns in it."""
import numpy as np
import pytest

from paper_1711_11418_gb300 import inputs as I
from paper_1711_11418_gb300 import vmc

pytestmark = pytest.mark.gpu


def problem(Np):
    p = I.make_problem("sr", I.chain(8, 1), 4, U=4.0, sub=(2, 1), jastrow="none", noise=0.1, seed=1)
    extra = np.random.default_rng(0).uniform(-1, 1, Np - 1 - p.n_f)
    return p.copy_with(n_f=Np - 1, params=np.concatenate([p.params, extra]))


def test_systems_of_a_batch_share_the_workspace():
    import torch

    sizes = [1024 - 40 * (k % 5) for k in range(20)]   # 20 systems, streams shared by two or three
    rows = 4096
    rng = np.random.default_rng(3)
    base = rng.standard_normal((rows, 1024))
    E = rng.standard_normal(rows)
    with vmc.Context([problem(n) for n in sizes], rows // 4, seed=1, precision=vmc.FP64, max_samples=4) as ctx:
        for s, n in enumerate(sizes):
            ctx.set_samples(E, np.roll(base, 97 * s, axis=0)[:, :n], s)
        before = torch.cuda.mem_get_info()[0]
        p0 = [ctx.get_params(s) for s in range(len(sizes))]
        ctx.sr_step_all(1.0, 0.1, 0.0, solver=vmc.CHOLESKY)
        held = before - torch.cuda.mem_get_info()[0]
        x = [p0[s] - ctx.get_params(s) for s in range(len(sizes))]
    digits = 7 * 1024 * rows * 2
    # per system S (8 Np^2) and vectors and partial sums of columns (below 8 MiB)
    per_system = 8 * 1024 ** 2 + (8 << 20)
    assert held <= 8 * digits + len(sizes) * per_system + (32 << 20)
    for s, n in enumerate(sizes):
        O = np.roll(base, 97 * s, axis=0)[:, :n]
        X = O - O.mean(0)
        S = X.T @ X / rows
        S[np.diag_indices(n)] *= 1.1
        ref = np.linalg.solve(S, X.T @ (E - E.mean()) / rows)
        # condition below 40, sums of 4096 terms, parameters of order 1
        assert np.abs(x[s] - ref).max() <= 1e-12 * np.abs(ref).max() + 4 * 2.3e-16 * (1 + np.abs(p0[s]).max())


def test_workspace_grows_with_the_largest_system():
    """A small system first, then a larger one, then the small one again."""
    rng = np.random.default_rng(4)
    rows = 512
    sizes = [40, 300]
    O = [rng.standard_normal((rows, n)) for n in sizes]
    E = rng.standard_normal(rows)
    with vmc.Context([problem(n) for n in sizes], rows, seed=1, precision=vmc.FP64) as ctx:
        for s in range(2):
            ctx.set_samples(E, O[s], s)
        got = [ctx.get_sr_matrices(system=s)[0] for s in (0, 1, 0)]
        ctx.sr_step_all(0.1, 0.1, 0.0, solver=vmc.CHOLESKY)
        got.append(ctx.get_sr_matrices(system=1)[0])
    for S, s in zip(got, (0, 1, 0, 1)):
        X = O[s] - O[s].mean(0)
        ref = X.T @ X / rows
        assert np.abs(S - ref).max() <= 4 * rows * 2.3e-16 * np.abs(np.diag(ref)).max()
