"""The FP64 force paths (md_forces of an FP64 system and md_forces_noalloc) on inputs that their FP32 tests and
bit-pattern comparisons have to carry: positions that are not numbers, particles in one place, any unit of length."""
import numpy as np
import pytest

import oracle
from paper_2001_07089_gb300 import kamd
from paper_2001_07089_gb300 import workloads as wl
from tests.helpers import force_errors, ka_params, melted

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    kamd.load()


def noalloc(pos, types, L, eps=wl.KA_EPS, sig=wl.KA_SIG, rc=wl.KA_RC):
    import torch
    n = len(pos)
    f = torch.empty((n, 3), dtype=torch.float64, device="cuda")
    e = torch.empty(2, dtype=torch.float64, device="cuda")
    dpos = torch.tensor(pos, dtype=torch.float64, device="cuda")
    dtyp = torch.tensor(np.asarray(types, dtype=np.uint8), device="cuda")
    torch.cuda.synchronize()
    kamd.md_forces_noalloc(n, dpos, dtyp, len(eps), L, eps, sig, rc, f, e[:1], e[1:],
                           torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    return f.cpu().numpy(), float(e[0]), float(e[1])


@pytest.mark.parametrize("bad", [np.nan, -np.nan, np.inf, -np.inf], ids=["nan", "-nan", "inf", "-inf"])
def test_a_particle_without_a_position_acts_on_none(bad):
    """It takes part in no pair: its force is zero, the others' and the energy are those without it, also
    after steps, and it crosses no box edge."""
    pos, vel, types, L = melted(1000, 22, nsteps=200)
    pos, rest = pos.copy(), np.arange(1000) != 7
    pos[7, 0] = bad
    f_ref, pe_ref, _ = oracle.forces(pos[rest], types[rest], ka_params(), L)
    f, pe, _ = noalloc(pos, types, L)
    assert np.all(f[7] == 0.0) and force_errors(f[rest], f_ref)[0] <= 1e-12
    assert abs(pe - pe_ref) <= 1e-12 * abs(pe_ref)
    with kamd.System(1000, L, types, wl.KA_EPS, wl.KA_SIG, wl.KA_RC, 1.0, 0.3, "fp64") as s:
        s.set_state(pos, vel)
        f, pe, _ = s.forces()
        assert np.all(f[7] == 0.0) and force_errors(f[rest], f_ref)[0] <= 1e-12
        assert abs(pe[0] - pe_ref) <= 1e-12 * abs(pe_ref)
        s.step_nve(0.002, 10)
        p, _, img = s.get_state()
        f, _, _ = s.forces()
    assert img[7, 0] == 0 and np.isnan(p[7, 0])
    f_ref, _, _ = oracle.forces(p[rest], types[rest], ka_params(), L)
    assert np.all(f[7] == 0.0) and force_errors(f[rest], f_ref)[0] <= 1e-12


def test_particles_in_one_place():
    """Two particles at the same point: infinite energy, forces that are not numbers on these two alone."""
    pos, _, types, L = melted(1000, 22, nsteps=200)
    pos = pos.copy()
    pos[9] = pos[400]
    two = np.isin(np.arange(1000), (9, 400))
    f_ref, _, _ = oracle.forces(pos[~two], types[~two], ka_params(), L)
    one, _, _ = oracle.forces(pos[np.arange(1000) != 9], types[np.arange(1000) != 9], ka_params(), L)
    other, _, _ = oracle.forces(pos[np.arange(1000) != 400], types[np.arange(1000) != 400], ka_params(), L)
    # every other particle feels both
    f_ref = np.delete(one, 399, axis=0) + np.delete(other, 9, axis=0) - f_ref
    with kamd.System(1000, L, types, wl.KA_EPS, wl.KA_SIG, wl.KA_RC, 1.0, 0.3, "fp64") as s:
        s.set_state(pos)
        f, pe, w = s.forces()
        results = [(f, pe[0], w[0]), noalloc(pos, types, L)]
    for f, pe, w in results:
        assert pe == np.inf and w == np.inf
        assert np.all(np.isnan(f[two])) and force_errors(f[~two], f_ref)[0] <= 1e-11


def test_autotune_names_the_lanes_that_run():
    """An FP64 system has at least four lanes per particle: fewer are the same program, and are not tried."""
    n = 256
    L = wl.box_length(n)
    with kamd.System(n, L, wl.ka_types(n, 3).astype(np.int32), wl.KA_EPS, wl.KA_SIG, wl.KA_RC, 1.0, 0.3, "fp64") as s:
        s.set_tuning(threads_per_atom=1, block_size=256, skin=0.3, skin_outer=0.3)
        s.init_lattice(0.5, seed=5)
        for skin in (None, 0.25):
            tun, _ = s.autotune(0.004, probe_steps=4, skin=skin)
            assert tun["threads_per_atom"] >= 4 and s.tuning["threads_per_atom"] >= 4, tun


@pytest.mark.parametrize("power", [-300, -70, -41, 41, 70, 300])
def test_any_unit_of_length(power):
    """Lengths in units of 2^power: their squares leave the range of FP32 (and sigma^12 that of FP64). Energies,
    virials and g(r) are those of power 0, forces and positions scale, in single calls and over steps."""
    pos, vel, types, L = melted(1000, 22, nsteps=200)
    f1, pe1, w1 = noalloc(pos, types, L)

    def run(u, skin):
        with kamd.System(1000, L * u, types, wl.KA_EPS, wl.KA_SIG * u, wl.KA_RC * u, u ** -2.0, skin, "fp64") as s:
            s.set_tuning(skin=skin, skin_outer=skin)
            s.set_state(pos * u, vel * u)
            f, pe, w = s.forces()
            log = s.step_nve(0.004, 20, log_every=10)
            g = s.rdf(0.02 * u, 200, reset=True)
            p, v, img = s.get_state()
            return f * u, pe, w, p / u, v / u, img, g, log["pe_per_n"], log["T"], s.count_pairs(), s.msd() / u ** 2

    u = 2.0 ** power
    f, pe, w = noalloc(pos * u, types, L * u, wl.KA_EPS, wl.KA_SIG * u, wl.KA_RC * u)
    assert force_errors(f * u, f1)[0] <= 1e-12 and abs(pe - pe1) <= 1e-12 * abs(pe1) and abs(w - w1) <= 1e-11 * abs(w1)
    # (a skin beyond 2 is refused, and a skin of 0.3 at large lengths is next to none)
    a, b = run(1.0, 0.3), run(u, 0.3 * min(u, 1.0))
    assert force_errors(b[0], a[0])[0] <= 1e-12
    for x, y in zip(b[1:], a[1:]):
        assert np.allclose(x, y, rtol=1e-9, atol=1e-9), (x, y)


def test_reciprocal_in_the_pair_term():
    """32 768 pairs alone in their cells, at r^2 over the cutoff's range and beside powers of two. With u = 2^-53:
    1/r^2 is off by at most 2 u (r^2 and the reciprocal rounded), its cube by 8 u, the two terms of the bracket
    by 16 + 6 and 8 + 5 u (sigma and epsilon are 1), the product with 1/r^2 and r by 4 u more."""
    n, L, cell = 32768, 256.0, 8.0
    rng = np.random.default_rng(12)
    r = rng.uniform(0.72, 2.49, n)
    near = np.sqrt(2.0 ** rng.integers(-1, 3, n // 4) * (1 + rng.integers(-8, 9, n // 4) * 2.0 ** -44))
    r[:n // 4] = np.clip(near, 0.72, 2.49)
    a = np.stack(np.unravel_index(np.arange(n), (32,) * 3), 1) * cell + 2.0
    axis = np.arange(n) % 3
    b = a.copy()
    b[np.arange(n), axis] += r
    d = (b - a)[np.arange(n), axis].astype(np.longdouble)  # exact: both are multiples of 2^-45
    one = np.ones((1, 1))
    f, _, _ = noalloc(np.concatenate([a, b]), np.zeros(2 * n), L, one, one, 2.5 * one)
    got = f[n + np.arange(n), axis].astype(np.longdouble)
    y = 1 / (d * d)
    attract, repel = 24 * y ** 3, 48 * y ** 6
    bound = 32 * np.longdouble(2) ** -53 * (repel + attract) * y * d
    assert np.all(np.abs(got - (repel - attract) * y * d) <= bound)
    assert np.array_equal(f[:n], -f[n:])
