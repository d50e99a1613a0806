"""The plain form's sweep at electron counts around its warps and powers of
two: its sums leave out the lanes and warps without electrons, and its hop
decisions are screened in FP32.  The same chain by batches of proposals, which
use full sums and the FP64 exponential throughout, has to come out: equal
configurations and counters, and local energies to 1e-9 (sums in another
order; cond(X) of sampled placements stays below 1e6)."""
import numpy as np
import pytest

from paper_1711_11418_gb300 import inputs as I
from paper_1711_11418_gb300 import vmc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Ns,N", [(4, 1), (6, 2), (8, 3), (9, 5), (40, 31), (40, 32), (41, 33),
                                  (80, 63), (90, 65), (160, 127), (160, 128)])
@pytest.mark.parametrize("scale", [0.1, 6.0])
def test_chain_equals_the_batched_one(Ns, N, scale):
    """scale: size of the Jastrow parameters; 6 brings factors beyond the
    range the screening decides."""
    p = I.make_problem("fs", I.chain(Ns, -1), 2 * N, U=3.0, f_full=True, jastrow="chain",
                       f_init="none", noise=0.0, p_exchange=0.4)
    rng = np.random.default_rng(Ns + 1000 * N)
    x = rng.uniform(-1.0, 1.0, p.params.size)
    x[:p.n_g + p.n_v] *= scale
    p = p.copy_with(params=x)
    cfg = I.initial_configs(Ns, 2 * N, 6, False, 3)
    out = []
    for batch in (1, 4):
        with vmc.Context(p, 6, seed=11, max_samples=2) as ctx:
            ctx.set_configs(cfg)
            ctx.set_proposal_batch(batch)
            ctx.sample(2, 2, 1)
            E, _ = ctx.get_samples(with_O=False)
            out.append((E, *ctx.get_configs()))
    (E1, ele1, ctr1), (E4, ele4, ctr4) = out
    np.testing.assert_array_equal(ele1, ele4)
    np.testing.assert_array_equal(ctr1, ctr4)
    np.testing.assert_allclose(E1, E4, rtol=1e-9, atol=1e-9 * max(1.0, np.abs(E4).max()))


def test_two_walkers_per_sm_equal_the_wide_layout():
    """16 x 16, N = 112: proposals one at a time take a walker of half an SM's
    shared memory, with the O rows accumulated in global memory; batches a
    larger one.  Same chain, E and O."""
    p = I.square16_hubbard()
    out = []
    for batch in (1, 4):
        with vmc.Context(p, 4, seed=5, max_samples=2) as ctx:
            ctx.set_proposal_batch(batch)
            ctx.sample(0, 2, 1)
            out.append((*ctx.get_samples(), *ctx.get_configs()))
    (E1, O1, ele1, ctr1), (E4, O4, ele4, ctr4) = out
    np.testing.assert_array_equal(ele1, ele4)
    np.testing.assert_array_equal(ctr1, ctr4)
    np.testing.assert_allclose(E1, E4, rtol=1e-9, atol=1e-9 * np.abs(E4).max())
    np.testing.assert_allclose(O1, O4, rtol=1e-9, atol=1e-9 * np.abs(O4).max())
