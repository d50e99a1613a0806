"""Pair correlations at the sizes where the kernel's tiling changes: electron
counts around 32, 64 and 128 (the columns a lane holds and the staged chunks),
no empty site, one electron per spin, more singly occupied sites than rows of
G_up fit shared memory, and walker counts around the occupation kernel's 256.
Reference: the oracle's local correlations on the same configurations.

Tolerances, as for the small models: 1e-10 of max(1, |reference|) in the plain
form; 1e-4 in the mixed form on configurations with cond(X) < 1e3; the
diagonal kinds exactly."""
import numpy as np
import pytest

from oracle import fock
from oracle.physics import local_correlation
from oracle.wavefunction import Wavefunction
from paper_1711_11418_gb300 import inputs as I
from paper_1711_11418_gb300 import vmc

pytestmark = pytest.mark.gpu


def problem(Ns, N):
    p = I.make_problem("cs", I.chain(Ns, -1), 2 * N, U=3.0, f_full=True, jastrow="chain",
                       f_init="none", noise=0.0, p_exchange=0.5)
    rng = np.random.default_rng(Ns + 1000 * N)
    x = rng.uniform(-1.0, 1.0, p.params.size)
    x[:p.n_g + p.n_v] *= 0.1
    return p.copy_with(params=x)


def draw(p, rng, apart):
    """A configuration; apart: the two spins on different sites."""
    Ns, N = p.Ns, p.Ne // 2
    if apart:
        return rng.permutation(Ns)[:2 * N].astype(np.int32)
    return np.concatenate([rng.permutation(Ns)[:N], rng.permutation(Ns)[:N]]).astype(np.int32)


@pytest.mark.parametrize("Ns,N,apart,precision", [
    (6, 1, False, vmc.FP64), (9, 9, False, vmc.MIXED), (33, 31, False, vmc.FP64),
    (40, 32, False, vmc.MIXED), (41, 33, False, vmc.FP64), (70, 64, False, vmc.FP64),
    (71, 65, False, vmc.MIXED), (100, 97, False, vmc.FP64), (256, 128, True, vmc.FP64),
    (256, 128, True, vmc.MIXED)])
def test_correlations_by_size(Ns, N, apart, precision):
    p = problem(Ns, N)
    wf = Wavefunction(p)
    rng = np.random.default_rng(5)
    cfg = []
    for _ in range(400):
        c = draw(p, rng, apart)
        if np.linalg.cond(wf.X(fock.from_labels(c, Ns))[0]) < 1e3:
            cfg.append(c)
            if len(cfg) == 2:
                break
    assert len(cfg) == 2
    cfg = np.array(cfg, np.int32)
    with vmc.Context(p, 2, seed=3, precision=precision) as ctx:
        ctx.set_configs(cfg)
        c = ctx.measure_corr()
    states = [fock.from_labels(e, Ns) for e in cfg]
    occ = np.zeros((2, 2, Ns), bool)
    for w, e in enumerate(cfg):
        occ[w, 0, e[:N]] = True
        occ[w, 1, e[N:]] = True
    entries = [(k, int(i), int(j)) for k in (0, 1, 4, 5) for i, j in rng.integers(0, Ns, (4, 2))]
    for w in range(2):
        up, dn = occ[w]
        pools = {0: (~up, up), 1: (~dn, dn), 4: (dn & ~up, up & ~dn)}
        for k, (a, b) in pools.items():
            a, b = np.flatnonzero(a), np.flatnonzero(b)
            if len(a) and len(b):
                # the ends of both lists, and pairs between
                pairs = [(a[0], b[0]), (a[-1], b[-1]), (a[0], b[-1]), (a[-1], b[0])]
                pairs += [(rng.choice(a), rng.choice(b)) for _ in range(8)]
                entries += [(k, int(i), int(j)) for i, j in pairs]
    tol = 1e-10 if precision == vmc.FP64 else 1e-4
    for k, i, j in entries:
        ref = 0.5 * sum(local_correlation(wf, s, k, i, j) for s in states)
        assert abs(c[k, i, j] - ref) <= tol * max(1.0, abs(ref)), (k, i, j, c[k, i, j], ref)


@pytest.mark.parametrize("Ns,W", [(31, 255), (33, 256), (64, 257)])
def test_occupation_counts_by_size(Ns, W):
    p = problem(Ns, 2)
    rng = np.random.default_rng(W)
    cfg = np.array([draw(p, rng, False) for _ in range(W)], np.int32)
    with vmc.Context(p, W, seed=3) as ctx:
        ctx.set_configs(cfg)
        c = ctx.measure_corr()
    up, dn = np.zeros((W, Ns)), np.zeros((W, Ns))
    for w, e in enumerate(cfg):
        up[w, e[:2]] = 1
        dn[w, e[2:]] = 1
    # integer sums times 1/W: one rounding of a product of two exact factors
    n, sz = up + dn, up - dn
    np.testing.assert_allclose(c[2], n.T @ n / W, rtol=0, atol=1e-15)
    np.testing.assert_allclose(c[3], 0.25 * (sz.T @ sz) / W, rtol=0, atol=1e-15)
