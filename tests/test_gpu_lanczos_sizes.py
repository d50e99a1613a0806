"""Power-Lanczos local values at the sizes where the kernel's tiling and
storage change: site counts around the tiles of its table products, and the
counts from which a warp's vectors no longer fit shared memory (FP64 and
FP32).  Reference: the oracle's F(x, H), F(x, H^2) by amplitudes."""
import numpy as np
import pytest

from oracle import fock
from oracle.lanczos import local_f
from oracle.wavefunction import Wavefunction
from paper_1711_11418_gb300 import inputs as I
from paper_1711_11418_gb300 import vmc

from helpers import condition_ok

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Ns,N,precision", [
    (17, 3, vmc.FP64), (63, 4, vmc.FP64), (65, 2, vmc.FP64), (127, 3, vmc.MIXED), (129, 2, vmc.FP64),
    (129, 3, vmc.MIXED), (1100, 2, vmc.FP64), (2200, 2, vmc.MIXED)])
def test_local_values_by_size(Ns, N, precision):
    p = I.make_problem("lz", I.chain(Ns, -1), 2 * N, U=3.0, t2=0.25, f_full=True, jastrow="none",
                       f_init="none", noise=0.0, p_exchange=0.5)
    rng = np.random.default_rng(Ns)
    params = rng.uniform(-1.0, 1.0, p.params.size)
    params[:p.n_g] = -0.3
    p = p.copy_with(params=params)
    wf = Wavefunction(p)
    cfg, s = [], 1
    while len(cfg) < 2:
        c = I.initial_configs(p.Ns, p.Ne, 1, False, s)[0]
        s += 1
        if condition_ok(wf, c):
            cfg.append(c)
    cfg = np.array(cfg, np.int32)
    with vmc.Context(p, 2, seed=3, precision=precision) as ctx:
        ctx.set_configs(cfg)
        f1, f2, _ = ctx.lanczos_moments()
    ref = np.array([local_f(wf, fock.from_labels(c, p.Ns)) for c in cfg])
    # FP64: the bound of the small models' test.  FP32: tables and ratios of
    # relative error cond * 2^-24 at most (cond(M) < 1e3 for small N), summed
    # over terms of both signs: 1e-4 of the largest value.
    tol = 1e-10 if precision == vmc.FP64 else 1e-4
    for got, want in ((f1, ref[:, 0]), (f2, ref[:, 1])):
        assert np.max(np.abs(got - want)) <= tol * max(1.0, np.max(np.abs(want)))
