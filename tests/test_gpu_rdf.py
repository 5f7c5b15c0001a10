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


def seconds(s, dr, nbins):
    import time
    best = np.inf
    for _ in range(4):
        t = time.perf_counter()
        s.rdf(dr, nbins, reset=True)
        best = min(best, time.perf_counter() - t)
    return best


def test_cost_follows_the_particles_not_the_cells():
    """10 000 particles in a box of 620 cells per edge cost what they do in one of 62: the pairs are far fewer,
    and walking the empty cells alone took 200 times as long."""
    n = 10000
    types = wl.ka_types(n, 6).astype(np.int32)
    t = []
    for L in (100.0, 1000.0):
        with system(n, L, types, "mixed") as s:
            s.set_state(wl.uniform_positions(n, L, 6))
            t.append(seconds(s, 0.01, 400))
    assert t[1] < 10 * t[0], t


def test_largest_replica_of_a_batch_gets_its_share_of_the_gpu():
    """120 000 particles and all pairs to L/2 cost about as much with 255 pairs of particles beside them as alone."""
    n, small = 120000, 255
    L = wl.box_length(n)
    types = wl.ka_types(n, 3).astype(np.int32)
    pos = np.concatenate([wl.uniform_positions(n, L, 3), wl.uniform_positions(2 * small, L, 4)])
    t, g = [], []
    for k in (0, small):
        m = n + 2 * k
        with system([n] + [2] * k if k else n, [L] * (k + 1) if k else L,
                    np.concatenate([types, np.tile(np.int32([0, 1]), k)]), "mixed") as s:
            s.set_state(pos[:m])
            t.append(seconds(s, 0.0499 * L, 10))
            g.append(s.rdf(0.0499 * L, 10, reset=True)[:2] * (k + 1))  # like pairs: the large replica's
    assert np.allclose(g[0], g[1], rtol=1e-12)
    assert t[1] < 10 * t[0], t


@pytest.mark.parametrize("ndim,L", [(3, 30.0), (3, 60.0), (2, 150.0)])
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_dilute_boxes_and_droplets(prec, ndim, L):
    """Half the particles anywhere in the box, half in a dense droplet on its corner: empty cells, cells with
    one particle, and runs of cells long enough to be cut, after steps that move particles from their cells."""
    n, m = 3000, {3: 14, 2: 50}[ndim]
    half = 0.5 * (n / 2) ** (1 / ndim)  # half the droplet's edge at number density 1
    k = int(np.ceil((n // 2) ** (1 / ndim)))
    site = np.stack(np.unravel_index(np.arange(n // 2), (k,) * ndim), 1)
    drop = (site + 0.5) * (2 * half / k) - half
    gas = (np.stack(np.unravel_index(np.arange(m ** ndim), (m,) * ndim), 1) + 0.5) * (L / m) - 0.5 * L
    gas = gas[np.any(np.abs(gas) > half + 1.5, axis=1)]
    gas = gas[np.random.default_rng(8).permutation(len(gas))[:n - n // 2]]
    gas += np.random.default_rng(9).uniform(-0.5, 0.5, gas.shape)
    pos = np.full((n, 3), 0.5 * L)
    pos[:, :ndim] = np.concatenate([drop, gas]) % L
    types = wl.ka_types(n, 8).astype(np.int32)
    dr, nbins = 0.02, 200
    with system(n, L, types, prec, ndim=ndim) as s:
        s.set_state(pos)
        s.step_nvt(0.002, 1, 0.5, kind=kamd.MD_NVT_RESAMPLE, param=1, seed=3)
        s.step_nve(0.002, 20)
        g = s.rdf(dr, nbins, reset=True)
        p, _, _ = s.get_state()
    ref = oracle.rdf(p, types, L, dr, nbins, ndim=ndim)
    k = np.arange(nbins)
    na = int(np.sum(types == 0))
    nb = n - na
    shell = 4 / 3 * np.pi * ((k + 1.0) ** 3 - k ** 3) * dr ** 3 if ndim == 3 else np.pi * (2 * k + 1.0) * dr ** 2
    w = np.outer([na * (na - 1.0), nb * (nb - 1.0), na * float(nb)], shell / L ** ndim)
    c, r = np.rint(g * w), np.rint(ref * w)
    assert r.sum() > 10 * n and np.max(np.abs(g * w - c)) < 1e-6
    assert np.array_equal(c, r)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_uneven_batch_many_bins_and_accumulation(prec):
    """Replicas of 6000, 20 and 700 particles, more bins than a CTA keeps counts for, after steps: the mean of the
    replicas' counts is the oracle's; a second call without reset leaves g(r) as it is, another dr starts anew."""
    ns = [6000, 20, 700]
    Ls = [wl.box_length(6000), 9.0, wl.box_length(700)]
    types = [wl.ka_types(n, 40 + k).astype(np.int32) for k, n in enumerate(ns)]
    off = np.concatenate([[0], np.cumsum(ns)])
    with system(ns, Ls, np.concatenate(types), prec) as s:
        s.init_lattice([1.0, 0.3, 2.0], seed=21)
        s.step_nve(0.004, 30)
        p, _, _ = s.get_state()
        for dr, nbins in ((0.0025, 1500), (0.01, 300), (0.005, 300)):
            g = s.rdf(dr, nbins, reset=(nbins > 300))
            ref = [oracle.rdf(p[off[k]:off[k + 1]], types[k], Ls[k], dr, nbins) for k in range(3)]
            assert np.allclose(g, np.mean(ref, axis=0), rtol=1e-12, atol=0)
            assert np.allclose(s.rdf(dr, nbins), g, rtol=1e-12, atol=0)


@pytest.mark.parametrize("n,L", [(1000, 9.4), (3000, 40.0)])
def test_a_particle_without_a_position_is_in_no_pair(n, L):
    """FP64: the 32-bit words of a position that is not a number are those of some place; no pair is counted there."""
    pos = wl.uniform_positions(n, L, 31)
    pos[:200] = np.random.default_rng(2).uniform(-1.0, 1.0, (200, 3)) % L  # close to where a NaN's words are
    pos[n // 2, 1] = np.nan
    types = wl.ka_types(n, 31).astype(np.int32)
    rest = np.arange(n) != n // 2
    dr, nbins = 0.02, 200
    with system(n, L, types, "fp64") as s:
        s.set_state(pos)
        g = s.rdf(dr, nbins, reset=True)
    ref = counts(oracle.rdf(pos[rest], types[rest], L, dr, nbins), types[rest], L, dr, nbins)
    assert np.array_equal(counts(g, types, L, dr, nbins), ref)
