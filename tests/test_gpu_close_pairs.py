"""FP64 forces of close pairs and of long boxes (one-species tables, whose pair terms are built from FP32
pieces over whole-number separations): isolated pairs 0.001 to 6 Å apart in boxes up to 30,000 Å long,
where the unit of the whole numbers grows.  Every pair's force is compared with the oracle's on its own,
at the relative error of 1/r that the FP64 precision states at any distance (4e-13): a force moves by
that share of its terms m through 1/r and of their radial sensitivities q and e through r, with a
quarter to spare; rho likewise."""
import numpy as np
import pytest

import oracle
from paper_1107_2619_gb300 import inputs as I, md

pytestmark = pytest.mark.gpu

EPS = 5e-13
R = np.array([0.001, 0.003, 0.01, 0.02, 0.03, 0.05, 0.07, 0.1, 0.2, 0.35, 0.5, 0.7, 0.95, 1.05, 1.5, 2.0, 2.5, 3.5, 6.0])


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1107_2619_gb300 import build
    build.build()


def dimers(length, r_min, fine):
    """One pair per distance, 20 Å apart along z and at random elsewhere.  Coarse coordinates (multiples
    of 2^-38, across the faces in x and y) have exact differences at every length; fine ones lie near the
    origin or anywhere else in a short box, off the whole-number unit."""
    g = np.random.default_rng(int(length) + fine)
    box = np.array([24.0, 24.0, length])
    z = np.linspace(3.0, length - 8.0, len(R)) if not fine else 1.0 + 20.0 * np.arange(len(R))
    d = g.normal(size=(len(R), 3))
    d *= (R / np.linalg.norm(d, axis=1))[:, None]
    if fine:
        a = np.stack([1.0 + g.uniform(0.0, 1.0, len(R)), 2.0 + g.uniform(0.0, 8.0, len(R)), z], axis=1)
        d = np.abs(d)
    else:
        a = np.stack([g.uniform(-0.4, 0.4, len(R)), g.uniform(0.0, 24.0, len(R)), z], axis=1)
    pos = np.concatenate([a, a + d])
    if not fine:
        pos = np.round(pos * 2.0 ** 38) / 2.0 ** 38
        pos[:, :2] = np.mod(pos[:, :2], 24.0)
    pot = I.sc_cu_tables(r_min=r_min)
    n = len(pos)
    return I.Workload(name="pairs", pos=pos, vel=np.zeros_like(pos), species=np.zeros(n, np.int32), box=box,
                      potential=pot, skin=0.3, k_max=16, dt_fs=0.0, steps=1, temperature=0.0)


def check_pair_forces(w, walk, lanes):
    ref = oracle.forces(w.pos, w.species, w.box, w.potential, skin=w.skin, k_max=w.k_max)
    sc = oracle.eam_error_scales(w.pos, w.species, w.box, w.potential, ref["count"], ref["list"], ref["dF"])
    bound = EPS * (2.0 * sc["m"] + sc["q"] + sc["e"])
    r = np.linalg.norm(np.mod(w.pos[len(w.pos) // 2:] - w.pos[:len(w.pos) // 2] + w.box / 2, w.box) - w.box / 2, axis=1)
    dphi = np.array([oracle.pair_value(w.potential, 1, 0, 0, x)[1] for x in r])
    rho_bound = EPS * (np.abs(ref["rho"]) + np.tile(r * np.abs(dphi), 2))
    with md.System(w, precision="fp64", passes=walk, lanes_per_atom=lanes) as s:
        s.eam_forces()
        assert np.array_equal(np.sort(s.neighbours()[0]), np.sort(ref["count"]))
        for step in (0, 1):   # the stand-alone passes, then the step kernel's (dt = 0: nothing moves)
            s.step(step)
            err = np.abs(s.forces() - ref["force"]).max(axis=1)
            assert np.all(err <= bound), (err / bound).reshape(2, -1).max(axis=0)
            rho = s.get(md.MD_GET_RHO)
            assert np.all(np.abs(rho - ref["rho"]) <= rho_bound)


WALKS = [("auto", 1), ("auto", 8), ("half", 2), ("half", 8)]


@pytest.mark.parametrize("walk,lanes", WALKS)
@pytest.mark.parametrize("length,r_min,fine", [(400.0, 1.0, False), (400.0, 0.05, True), (4100.0, 1.0, False),
                                               (10000.0, 0.3, False), (30000.0, 1.0, False), (30000.0, 1.0, True)])
def test_each_pair_force_at_any_distance(length, r_min, fine, walk, lanes):
    check_pair_forces(dimers(length, r_min, fine), walk, lanes)


@pytest.mark.parametrize("walk,lanes", WALKS)
def test_first_knot_near_the_cutoff(walk, lanes):
    """Tables from 5.8 to 6.2 Å: below the first knot the squares r^2 and rho_0^2 differ by more than half
    of what 64 bits hold."""
    w = dimers(400.0, 1.0, False)
    w.potential = I.sc_cu_tables(n_knots=500, lattice_a=3.1, r_min=5.8)
    check_pair_forces(w, walk, lanes)


@pytest.mark.parametrize("walk,lanes", [("auto", 4), ("half", 8)])
def test_steps_with_close_pairs(walk, lanes):
    """Several steps in one call, with scheduled rebuilds: the full list's force pass reads the positions of
    close pairs, so the next step opens after it.  Positions, of up to 400 Å, to a few units in the last
    place; velocities to the forces' bound, summed over the steps."""
    w = dimers(400.0, 1.0, False)
    steps = 7
    w.dt_fs = dt = 1e-3
    ref = oracle.run_vv(w.pos, w.vel, w.species, w.potential.masses, w.box, w.potential, dt, steps, w.skin, w.k_max,
                        rebuild_every=3)
    with md.System(w, precision="fp64", passes=walk, lanes_per_atom=lanes, rebuild_every=3) as s:
        s.step(steps)
        pos, vel = s.positions(), s.velocities()
    assert np.abs(pos - ref["pos"]).max() <= 4.0 * np.spacing(400.0)
    assert np.abs(vel - ref["vel"]).max() <= 100.0 * EPS * np.abs(ref["vel"]).max()


@pytest.mark.parametrize("walk,lanes", WALKS)
@pytest.mark.parametrize("n_knots,r_min", [(300, 1.3), (777, 1.7)])
def test_pairs_beside_a_knot(n_knots, r_min, walk, lanes):
    """Pairs between a knot and its FP32 value, which the row's interval must not be confused with: a
    cubic beside its interval has another slope."""
    w = dimers(1000.0, 1.0, False)
    w.potential = pot = I.sc_cu_tables(n_knots=n_knots, r_min=r_min)
    h = (pot.r_cut - r_min) / (n_knots - 1)
    k = np.arange(1, n_knots)
    knot = r_min + k * h
    rounded = (k * float(np.float32(h)) + float(np.float32(r_min))).astype(np.float32).astype(np.float64)
    pick = np.argsort(-np.abs(rounded - knot) * (knot < 3.0))[:40]   # the widest gaps
    z = np.linspace(3.0, 990.0, len(pick))
    a = np.stack([np.full(len(pick), 4.0), np.full(len(pick), 5.0), z], axis=1)
    a = np.round(a * 2.0 ** 38) / 2.0 ** 38
    b = a.copy()
    b[:, 0] += np.round(0.5 * (knot + rounded)[pick] * 2.0 ** 38) / 2.0 ** 38
    n = 2 * len(pick)
    w.pos, w.vel, w.species = np.concatenate([a, b]), np.zeros((n, 3)), np.zeros(n, np.int32)
    check_pair_forces(w, walk, lanes)


@pytest.mark.parametrize("walk,lanes", WALKS)
@pytest.mark.parametrize("length,fine", [(400.0, True), (30000.0, False)])
def test_energy_and_virial_with_close_pairs(length, fine, walk, lanes):
    """The close pairs' shares of E_i and of the virial (across the faces too) at the FP64 bar, by the
    stand-alone passes and by an energy step of the step kernel; two replicas in one batch give the same."""
    w = dimers(length, 1.0, fine)
    ref = oracle.forces(w.pos, w.species, w.box, w.potential, skin=w.skin, k_max=w.k_max)
    with md.System(w, precision="fp64", passes=walk, lanes_per_atom=lanes) as s:
        s.eam_forces()
        for step in (0, 1):
            s.step(step)
            e = s.energy()
            assert abs(e["pe"] - ref["pe"]) <= 1e-10 * abs(ref["pe"])
            assert np.abs(e["virial"] - ref["virial"]).max() <= 1e-10 * np.abs(ref["virial"]).max()
    with md.Batch([w, w], precision="fp64", passes=walk, lanes_per_atom=lanes) as b:
        b.eam_forces()
        f = b.forces()
    sc = oracle.eam_error_scales(w.pos, w.species, w.box, w.potential, ref["count"], ref["list"], ref["dF"])
    bound = EPS * (2.0 * sc["m"] + sc["q"] + sc["e"])
    assert np.all(np.abs(f - np.tile(ref["force"], (2, 1))).max(axis=1) <= np.tile(bound, 2))


@pytest.mark.parametrize("walk,lanes", [("auto", 4), ("half", 8)])
@pytest.mark.parametrize("kind", ["pc3", "nvt", "strain"])
def test_other_motions_with_close_pairs(kind, walk, lanes):
    """As test_steps_with_close_pairs, for the predictor-corrector, the thermostat and the strain ramp."""
    w = dimers(400.0, 1.0, False)
    steps = 7
    w.dt_fs = dt = 1e-3
    w.vel = np.random.default_rng(5).normal(0.0, 1e-4, w.pos.shape)
    args = (w.pos, w.vel, w.species, w.potential.masses, w.box, w.potential, dt, steps, w.skin, w.k_max)
    if kind == "strain":
        w.strain_rate_zz = -1.0e9
    with md.System(w, precision="fp64", passes=walk, lanes_per_atom=lanes,
                   integrator="pc3" if kind == "pc3" else "verlet") as s:
        if kind == "pc3":
            ref = oracle.run_pc3(*args)
        elif kind == "nvt":
            s.set_thermostat(300.0, tau_fs=20.0)
            s.eam_forces()
            ref = oracle.run_nvt(*args, 300.0, s.thermostat()[0, 2])
        else:
            ref = oracle.run_vv(*args, strain_rate_zz=w.strain_rate_zz)
        s.step(steps)
        pos, vel = s.positions(), s.velocities()
    assert np.abs(pos - ref["pos"]).max() <= 4.0 * np.spacing(400.0)
    assert np.abs(vel - ref["vel"]).max() <= 100.0 * EPS * np.abs(ref["vel"]).max()
