"""Contexts of different sizes side by side: making and using a small one must
not take shared memory from the kernels of a large one, in turn or from
another thread."""
import threading

import numpy as np
import pytest

from paper_1711_11418_gb300 import inputs as I
from paper_1711_11418_gb300 import vmc

pytestmark = pytest.mark.gpu


def hubbard(Lx, Ly, N, seed=1):
    p = I.make_problem("h", I.square(Lx, Ly, -1, -1), 2 * N, U=4.0, sub=(2, 2), jastrow="distance",
                       f_init="none", noise=0.5, seed=seed)
    p.params[:p.n_g + p.n_v] = -0.1
    return p


def gradient(ctx, p):
    ctx.set_params(p.params)
    ctx.sample(0, 1, 0)
    return ctx.get_samples()[0], ctx.get_sr_matrices(with_S=False)[1]


@pytest.mark.parametrize("precision", [vmc.FP64, vmc.MIXED])
@pytest.mark.parametrize("walkers", [8, 200])
def test_rebuilds_after_a_small_context_was_made(precision, walkers):
    big, small = hubbard(16, 16, 112), hubbard(4, 4, 2)
    with vmc.Context(big, walkers, seed=2, precision=precision) as a:
        E0, g0 = gradient(a, big)
        with vmc.Context(small, 4, seed=2, precision=precision) as b:
            gradient(b, small)
            E1, g1 = gradient(a, big)
            h0 = a.lanczos_moments()[0]
            b.lanczos_moments()
            h1 = a.lanczos_moments()[0]
    assert np.array_equal(E0, E1)
    assert np.allclose(g0, g1, rtol=1e-6, atol=1e-6 * np.abs(g0).max())   # O by atomic adds
    assert np.array_equal(h0, h1)


@pytest.mark.parametrize("precision", [vmc.FP64, vmc.MIXED])
def test_projected_rebuilds_after_a_small_projected_context(precision):
    big, small = hubbard(12, 12, 60), hubbard(4, 4, 2)
    ident = lambda p: (np.arange(p.Ns, dtype=np.int32)[None, :], np.ones((1, p.Ns), np.int8), np.ones(1))  # noqa: E731
    with vmc.Context(big, 8, seed=2, precision=precision) as a:
        a.set_projection(*ident(big))
        E0, _ = gradient(a, big)
        with vmc.Context(small, 4, seed=2, precision=precision) as b:
            b.set_projection(*ident(small))
            gradient(b, small)
            E1, _ = gradient(a, big)
    assert np.array_equal(E0, E1)


def test_power_lanczos_from_two_threads():
    """Two contexts of different sizes, each used by its own thread."""
    probs = [hubbard(12, 12, 60), hubbard(4, 4, 2)]
    errors, out = [], [[], []]
    ctxs = [vmc.Context(p, 16, seed=2, precision=vmc.MIXED) for p in probs]

    def work(k):
        try:
            for _ in range(100):
                out[k].append(ctxs[k].lanczos_moments()[0])
        except vmc.VmcError as e:
            errors.append((k, e))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for c in ctxs:
        c.close()
    assert not errors
    for k in range(2):
        assert all(np.array_equal(x, out[k][0]) for x in out[k])


@pytest.mark.parametrize("precision", [vmc.FP64, vmc.MIXED])
def test_placements_redrawn_on_the_contexts_stream(precision):
    """A third of the random placements are singular and drawn again, on a stream
    that does not wait for the default one: inverses and sites belong together."""
    import torch

    p = I.make_problem("redraw", I.square(8, 8), 6, sub=(1, 1), f_full=True, f_init="none", noise=0.0)
    f = np.random.default_rng(1).standard_normal((p.Ns, p.Ns))
    f[:8] = 0.0
    params = p.params.copy()
    params[p.n_g + p.n_v:] = f.reshape(-1)
    W = 3000
    st = torch.cuda.Stream()
    with vmc.Context(p.copy_with(params=params), W, seed=9, precision=precision, stream=st.cuda_stream) as ctx:
        ele, _ = ctx.get_configs()
        assert ele[:, :3].min() >= 8
        for w in range(0, W, 50):
            X = ctx.get_inverse(w)[0]
            M = f[np.ix_(ele[w, :3], ele[w, 3:])]
            assert np.abs(X @ M - np.eye(3)).max() <= 1e-12 * np.linalg.cond(M)
