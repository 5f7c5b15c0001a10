"""List builds and the FP64 force phase at the places where they can go wrong: entry queues that fill up
before a list ends, and lists built inside a run (after force phases of the same launch)."""
import numpy as np
import pytest

import oracle
from paper_2001_07089_gb300 import kamd
from paper_2001_07089_gb300 import workloads as wl
from tests.helpers import force_errors, melted

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    kamd.load()


@pytest.mark.parametrize("tpa", [1, 4, 8])
@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("mixed", 1e-5)])
def test_more_partners_than_a_queue_holds(prec, tol, tpa):
    """One species with a cutoff of 4.5 in the melted N = 1000 liquid: about 460 partners per particle,
    several times what the FP64 path's per-particle queues hold at once (128 or 256 entries)."""
    pos, _, _, L = melted(1000, 22, nsteps=200)
    types = np.zeros(1000, dtype=np.int32)
    eps, sig, rc = np.array([[1.0]]), np.array([[0.9]]), np.array([[4.5]])
    f_ref, v_ref, _ = oracle.forces(pos, types, oracle.Params(eps, sig, rc, 1.0), L)
    with kamd.System(1000, L, types, eps, sig, rc, 1.0, 0.1, prec) as s:
        s.set_tuning(threads_per_atom=tpa, skin=0.1, skin_outer=0.2)
        s.set_state(pos)
        f, pe, _ = s.forces()
        entries = s.info()["list_entries"]
    assert entries > 1000 * 400
    emax, e2 = force_errors(f, f_ref)
    assert emax <= tol and e2 <= tol, (emax, e2)
    assert abs(pe[0] - v_ref) <= max(tol, 1e-6 if prec == "mixed" else 0) * abs(v_ref)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("tpa,block", [(1, 512), (4, 256), (8, 256)])
def test_lists_built_in_a_run_equal_fresh_ones(prec, tpa, block):
    """With a skin so small that every step rebuilds, the list of the last step belongs to the final
    positions: a new system at those positions has as many candidate pairs, of either species."""
    pos, vel, types, L = melted(1000, 24, nsteps=200)
    counts = []
    with kamd.System(1000, L, types, wl.KA_EPS, wl.KA_SIG, wl.KA_RC, 1.0, 0.3, prec) as s:
        s.set_tuning(threads_per_atom=tpa, block_size=block, skin=0.01, skin_outer=0.01)
        s.set_state(pos, vel)
        s.step_nve(0.005, 6)
        info = s.info()
        assert info["rebuilds"] >= 6
        counts.append(info["list_entries"])
        p, v, _ = s.get_state()
    with kamd.System(1000, L, types, wl.KA_EPS, wl.KA_SIG, wl.KA_RC, 1.0, 0.3, prec) as s:
        s.set_tuning(threads_per_atom=tpa, block_size=block, skin=0.01, skin_outer=0.01)
        s.set_state(p, v)
        s.forces()
        counts.append(s.info()["list_entries"])
    # positions that pass through doubles may move a pair at the very edge of the radius
    assert abs(counts[0] - counts[1]) <= 2, counts


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("block", [128, 512])
def test_partial_rebuilds_of_more_replicas_than_threads(prec, block):
    """Replicas with and without cells, cold and hot, so that some rebuild while their neighbours do not;
    at block 128 there are more of them than a CTA has threads. Each is bitwise its stand-alone run."""
    sizes, temps = [250, 1000, 300, 2000, 500], [0.05, 3.0, 1.0, 0.3, 0.05, 2.0, 0.6]
    ns = [sizes[k % 5] for k in range(150)]
    Ts = [temps[k % 7] for k in range(150)]
    Ls = [wl.box_length(n) for n in ns]
    types = [wl.ka_types(n, 5 + k).astype(np.int32) for k, n in enumerate(ns)]
    tun = dict(threads_per_atom=4, block_size=block, skin=0.3, skin_outer=0.3)

    def run(n, L, t, T):
        with kamd.System(n, L, t, wl.KA_EPS, wl.KA_SIG, wl.KA_RC, 1.0, 0.3, prec) as s:
            s.set_tuning(**tun)
            s.init_lattice(T, seed=9)
            s.step_nve(0.004, 40)
            return s.get_state(), s.info()["rebuilds"]

    (p, v, img), rebuilds = run(ns, Ls, np.concatenate(types), Ts)
    assert rebuilds < 150 * 40
    off = np.concatenate([[0], np.cumsum(ns)])
    for k in (0, 1, 2, 3, 4, 71, 126, 127, 128, 129, 148, 149):
        (q, w, j), _ = run(ns[k], Ls[k], types[k], Ts[k])
        at = slice(off[k], off[k + 1])
        assert np.array_equal(q, p[at]) and np.array_equal(w, v[at]) and np.array_equal(j, img[at]), k


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_few_replicas_rebuilding_together_equal_their_own_runs(prec):
    """Eight replicas have more list-build groups than there are SMs but work enough for one CTA per SM: short
    launches that begin with all their rebuilds take more CTAs, long ones do not. Both are bitwise the same."""
    n, nrep, L = 1000, 8, wl.box_length(1000)
    types = [wl.ka_types(n, 30 + k).astype(np.int32) for k in range(nrep)]

    def run(k, cuts):
        t = np.concatenate(types) if k is None else types[k]
        m = nrep if k is None else 1
        with kamd.System([n] * m if m > 1 else n, [L] * m if m > 1 else L, t, wl.KA_EPS, wl.KA_SIG, wl.KA_RC, 1.0, 0.3,
                         prec) as s:
            s.init_lattice([1.2] * m if m > 1 else 1.2, seed=19)
            f = s.forces()[0]
            for c in cuts:
                p, v, _ = s.get_state()
                s.set_state(p, v)  # (every replica rebuilds)
                s.step_nve(0.004, c)
            return s.get_state()[:2] + (f, s.forces()[0])

    for cuts in ((8, 60, 8, 60), (60, 8)):
        x = run(None, cuts)
        for k in (0, 3, 7):
            y = run(k, cuts)
            assert all(np.array_equal(a, b[k * n:(k + 1) * n]) for a, b in zip(y, x)), (cuts, k)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_thousands_of_replicas_equal_their_own_runs(prec):
    """2500 replicas, some with cells and some without, cold and hot, so that any of them rebuild together:
    each is found among the others (bitwise its stand-alone run), and their energies come back."""
    ns = [[30, 2, 64, 9, 100, 5, 40][k % 7] for k in range(2500)]
    Ls = [[6.0, 12.0, 8.0][k % 3] for k in range(2500)]
    Ts = [[0.01, 4.0, 0.5, 1.0, 0.1][k % 5] for k in range(2500)]
    types = [np.arange(n, dtype=np.int32) % 2 for n in ns]
    tun = dict(threads_per_atom=4, block_size=256, skin=0.2, skin_outer=0.2)

    def run(n, L, t, T):
        with kamd.System(n, L, t, wl.KA_EPS, wl.KA_SIG, wl.KA_RC, 1.0, 0.3, prec) as s:
            s.set_tuning(**tun)
            s.init_lattice(T, seed=17)
            s.step_nve(0.003, 30)
            f, pe, w = s.forces()
            return s.get_state() + (f,), np.stack([pe, w]), s.info()["rebuilds"]

    x, e, rebuilds = run(ns, Ls, np.concatenate(types), Ts)
    assert 2 * 2500 < rebuilds < 2500 * 30
    off = np.concatenate([[0], np.cumsum(ns)])
    for k in (0, 1, 2, 3, 30, 31, 32, 78, 79, 80, 511, 1023, 1024, 1025, 2448, 2498, 2499):
        y, d, _ = run(ns[k], Ls[k], types[k], Ts[k])
        assert all(np.array_equal(a, b[off[k]:off[k + 1]]) for a, b in zip(y, x)), k
        assert np.array_equal(d[:, 0], e[:, k]), k


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("kind", [kamd.MD_NVT_NOSE_HOOVER, kamd.MD_NVT_NOSE_HOOVER_EXACT], ids=["nh", "nh-exact"])
@pytest.mark.parametrize("n,tpa", [(250, 8), (1000, 1), (32768, 4), (32800, 2)])
def test_one_replica_under_nose_hoover_equals_a_batch_member(prec, kind, n, tpa):
    """Bitwise the same alone and in a batch, with the sums added in one level (up to 32768 particles) and
    in two, and whether a step also forms the potential energy (log_every=1) or the kinetic energy alone."""
    L = wl.box_length(n)
    types = wl.ka_types(n, 3).astype(np.int32)

    def run(nrep, log_every):
        Ts = [1.3, 0.7][:nrep]
        with kamd.System([n] * nrep if nrep > 1 else n, [L] * nrep if nrep > 1 else L, np.concatenate([types] * nrep),
                         wl.KA_EPS, wl.KA_SIG, wl.KA_RC, 1.0, 0.3, prec) as s:
            s.set_tuning(threads_per_atom=tpa, block_size=256, skin=0.3, skin_outer=0.6)
            s.init_lattice(Ts if nrep > 1 else Ts[0], seed=11)
            log = np.concatenate([s.step_nvt(0.004, 12, Ts if nrep > 1 else Ts[0], kind=kind, param=0.4,
                                             log_every=log_every) for _ in range(2)])
            return [x[:n] for x in s.get_state()], log[:, 0]

    a, la = run(1, 4)
    for b, lb in (run(2, 4), run(1, 1)):
        assert all(np.array_equal(x, y) for x, y in zip(a, b))
        last = lb if len(lb) == len(la) else lb[3::4]
        assert all(np.array_equal(la[f], last[f]) for f in la.dtype.names if f != "step")
    assert np.all(np.isfinite(la["T"])) and np.all(la["T"] > 0)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_planar_batch_of_unequal_groups_equals_its_members(prec):
    """Replicas in a plane at three densities: their list-build groups have unequal numbers of rows, and the
    groups off the plane are empty, so a CTA passes from an empty group to one of another shape. Each replica
    is bitwise its stand-alone run."""
    ns = [[400, 90, 900, 60, 250][k % 5] for k in range(40)]
    rho = [[1.2, 0.1, 0.6][k % 3] for k in range(40)]
    Ts = [[0.1, 1.5, 0.4, 0.8][k % 4] for k in range(40)]
    Ls = [float(np.sqrt(n / d)) for n, d in zip(ns, rho)]
    types = [wl.ka_types(n, 7 + k).astype(np.int32) for k, n in enumerate(ns)]

    def run(n, L, t, T):
        with kamd.System(n, L, t, wl.KA_EPS, wl.KA_SIG, wl.KA_RC, 1.0, 0.3, prec, ndim=2) as s:
            s.set_tuning(threads_per_atom=8, block_size=256, skin=0.3, skin_outer=0.3)
            s.init_lattice(T, seed=13)
            s.step_nve(0.004, 60)
            return s.get_state()

    p, v, img = run(ns, Ls, np.concatenate(types), Ts)
    off = np.concatenate([[0], np.cumsum(ns)])
    for k in (0, 1, 2, 3, 4, 5, 17, 38, 39):
        q, w, j = run(ns[k], Ls[k], types[k], Ts[k])
        at = slice(off[k], off[k + 1])
        assert np.array_equal(q, p[at]) and np.array_equal(w, v[at]) and np.array_equal(j, img[at]), k


def test_two_replicas_of_the_most_cells():
    """Two boxes of 1024 cells per edge hold 2^31 cells between them, one more than 31 bits count. Each
    replica's forces are the oracle's, and so after steps with rebuilds in between."""
    import torch
    if torch.cuda.mem_get_info()[0] < 60 << 30:
        pytest.skip("needs 60 GB of device memory")
    n, L = 60, 1700.0
    pos, vel, types, _ = melted(250, 21, nsteps=200)
    rng = np.random.default_rng(6)
    # clusters of particles from a melt, each somewhere in its box
    near = np.argsort(np.sum((pos - pos[0] - 1e-9) ** 2, axis=1))[:n]
    ps = [(pos[near] - pos[0] + rng.uniform(0, L, 3)) % L for _ in range(2)]
    t = types[near]
    with kamd.System([n, n], [L, L], np.concatenate([t, t]), wl.KA_EPS, wl.KA_SIG, wl.KA_RC, 1.0, 0.3, "mixed") as s:
        s.set_tuning(threads_per_atom=4, block_size=256, skin=0.2, skin_outer=0.2)
        s.set_state(np.concatenate(ps), np.concatenate([vel[near], -vel[near]]))
        f = [s.forces()[0]]
        s.step_nve(0.002, 40)
        f.append(s.forces()[0])
        p, _, _ = s.get_state()
        assert s.info()["rebuilds"] > 2
    for q, g in zip((np.concatenate(ps), p), f):
        for k in range(2):
            at = slice(k * n, (k + 1) * n)
            ref, _, _ = oracle.forces(q[at], t, oracle.Params(wl.KA_EPS, wl.KA_SIG, wl.KA_RC, 1.0), L)
            assert force_errors(g[at], ref)[0] <= 1e-4
