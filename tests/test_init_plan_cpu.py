"""The launch plan of the from-scratch inverses (host arithmetic, no GPU): the
shared memory it asks for holds the layout of the form it launches, for every
system of the context, on large lattices with few electrons as well."""
import ctypes as C
import itertools

import pytest

BLOCKED, STEPS, DF = 0, 1, 2
SMS = 152


class Plan(C.Structure):
    _fields_ = [("form", C.c_int), ("threads", C.c_int), ("smem", C.c_size_t)]


@pytest.fixture(scope="module")
def lib():
    from paper_1711_11418_gb300 import build
    L = C.CDLL(build.build())
    L.vmc_init_plan.restype = None
    L.vmc_init_smem.restype = C.c_size_t
    return L


def plan(lib, precision, df, exchange, N, Ns, work):
    out = Plan()
    n = len(N)
    lib.vmc_init_plan(precision, df, exchange, n, (C.c_int * n)(*N), (C.c_int * n)(*Ns), work, SMS,
                      C.byref(out))
    return out


def up(x, a):
    return -(-x // a) * a


def need(form, N, Ns):
    """Bytes the kernel's layout takes: matrix, scratch, 2 N sites and N rows."""
    pad = up(N, 16)
    matrix = pad * pad * 8 if form == BLOCKED else up(N * (N | 1) * 8, 16)
    scratch = up(4 * (2 * Ns + 1), 16)
    if form == BLOCKED:
        scratch = max(scratch, 7168)
        # a matrix close to singular is eliminated again with rows of odd stride,
        # whose end reaches into the scratch, the second elimination's state behind it
        assert N * (N | 1) * 8 <= matrix + 1024
    return matrix + scratch + 12 * N


def sizes(N):
    return sorted({max(N, 2), N + 1, 64, 144, 256, 831, 847, 848, 849, 863, 864, 865, 895, 896, 897, 1024, 4095, 4096}
                  - set(range(N)))


@pytest.mark.parametrize("precision,df,exchange", [(0, 0, 0), (0, 0, 1), (1, 0, 0), (1, 0, 1), (1, 1, 0)])
def test_shared_memory_holds_the_form_launched(lib, precision, df, exchange):
    for N in range(1, 129):
        for Ns, work in itertools.product(sizes(N), (1, SMS - 1, SMS, SMS + 1, 4 * SMS, 4 * SMS + 1, 5000)):
            p = plan(lib, precision, df, exchange, [N], [Ns], work)
            assert p.smem >= need(p.form, N, Ns), (N, Ns, work, p.form)
            assert p.smem <= 227 * 1024
            assert p.threads % 32 == 0 and 64 <= p.threads <= 256
            if p.form == BLOCKED:   # a warp per 16 rows and a thread per row
                assert p.threads >= 2 * up(N, 16)


def test_small_walker_counts_on_large_lattices(lib):
    """N = 32 and 48, where rows of odd stride are longer than the padded matrix."""
    for N, Ns in ((32, 864), (32, 1024), (32, 4096), (48, 848), (48, 1024), (48, 4096)):
        p = plan(lib, 0, 0, 0, [N], [Ns], 4)
        assert p.form == STEPS and p.smem == lib.vmc_init_smem(N, Ns, STEPS) == need(STEPS, N, Ns)
        assert lib.vmc_init_smem(N, Ns, BLOCKED) < need(STEPS, N, Ns)


def test_every_system_of_a_batch_fits(lib):
    systems = [(16, 4096), (48, 144), (32, 1024), (25, 2000), (1, 2), (47, 900)]
    for k in range(1, len(systems) + 1):
        for sub in itertools.combinations(systems, k):
            for work in (k, SMS, SMS + 1, 64 * k):
                p = plan(lib, 0, 0, 0, [s[0] for s in sub], [s[1] for s in sub], work)
                assert all(p.smem >= need(p.form, *s) for s in sub)
