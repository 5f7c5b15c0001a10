"""The g(r) histogram at the places where its counts could go wrong: large counts, each way of finding the
pairs, batches. Counts are whole numbers: they are compared exactly."""
import numpy as np
import pytest

import oracle
from paper_2001_07089_gb300 import kamd
from paper_2001_07089_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    kamd.load()


def system(n, L, types, prec, **kw):
    return kamd.System(n, L, types, wl.KA_EPS, wl.KA_SIG, wl.KA_RC, 1.0, 0.3, prec, **kw)


def weights(types, L, dr, nbins):
    """What turns g (3, nbins) into the counts behind it (like pairs twice)."""
    nb = int(np.sum(types))
    na = len(types) - nb
    k = np.arange(nbins)
    shell = 4.0 / 3.0 * np.pi * ((k + 1.0) ** 3 - k ** 3) * dr ** 3 / L ** 3
    return np.outer([na * (na - 1.0), nb * (nb - 1.0), na * float(nb)], shell)


def counts(g, types, L, dr, nbins):
    h = g * weights(types, L, dr, nbins)
    c = np.rint(h)
    assert np.max(np.abs(h - c)) < 1e-6 * max(1.0, c.max() * 1e-6)
    return c.astype(np.int64)


def test_counts_beyond_32_bits():
    """One replica of 120 000 particles among 1215 of two: 4.8e9 ordered AA pairs lie within L/2. They are
    counted in one bin as in 64, whose counts are all below 2^32."""
    n, small = 120000, 1215
    L = wl.box_length(n)
    types = wl.ka_types(n, 3).astype(np.int32)
    pos = np.concatenate([wl.uniform_positions(n, L, 3), wl.uniform_positions(2 * small, L, 4)])
    with system([n] + [2] * small, [L] * (small + 1), np.concatenate([types, np.tile(np.int32([0, 1]), small)]),
                "mixed") as s:
        s.set_state(pos)
        rmax = 0.499 * L
        one = s.rdf(rmax, 1, reset=True)
        many = s.rdf(rmax / 64, 64, reset=True)
    a = one * weights(types, L, rmax, 1)
    b = many * weights(types, L, rmax / 64, 64)
    # g is the mean over the replicas, of which the small ones have AB pairs only
    assert a[0, 0] * (small + 1) > 2.0 ** 32
    assert np.allclose(a[:, 0], b.sum(1), rtol=1e-12, atol=0)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_long_rows_count_as_the_oracle(prec):
    """All pairs of N = 16 400 to L/2: a warp bins more pairs than it holds between two moves of its counts."""
    n, nbins = 16400, 5
    L = wl.box_length(n)
    types = wl.ka_types(n, 5).astype(np.int32)
    pos = wl.uniform_positions(n, L, 5)
    dr = 0.4999 * L / nbins
    with system(n, L, types, prec) as s:
        s.set_state(pos)
        g = s.rdf(dr, nbins, reset=True)
        p, _, _ = s.get_state()
    ref = counts(oracle.rdf(p, types, L, dr, nbins), types, L, dr, nbins)
    assert np.array_equal(counts(g, types, L, dr, nbins), ref)
