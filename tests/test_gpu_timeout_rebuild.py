"""A stand-alone list rebuild whose grid barrier gives up (one block withholds its arrival; the others' wait
is bounded and short): the call reports the timeout, the passes behind it read no half-built list, no atom
is lost or moved, and the next call rebuilds and gives what a fresh context gives.  At every barrier of
the rebuild, as a context's first build and between steps."""
import numpy as np
import pytest

from paper_1107_2619_gb300 import inputs as I, md

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1107_2619_gb300 import build
    build.build()


def make(kind):
    if kind == "surrogate":
        theta = I.sur_init_weights(4).astype(np.float32)
        return md.SurrogateSystem(I.bcc_fe(9, seed=5), theta, np.ones(32, np.float32), np.full(32, 0.5, np.float32))
    w = I.fcc_cu(10, seed=3, sigma=0.05, n_knots=1000)   # 4,000 atoms: several blocks
    w.vel = w.vel * 3.0
    prec, walk = kind.split("-")
    return md.System(w, precision=prec, passes=walk)


KINDS = ["fp64-half", "fp64-list", "mixed-list", "df-list", "surrogate"]
BARRIERS = [(k, b) for k in KINDS for b in range(1, 11) if b != 9 or k == "fp64-half"]
_fresh = {}


def fresh(kind):
    """Forces at the start and the state after two calls of steps, with a rebuild and a force evaluation
    between them, as the recovering context makes (FP32 copies lie in the image of the last build)."""
    if kind not in _fresh:
        with make(kind) as s:
            s.eam_forces()
            f0 = s.forces()
            s.step(3)
            s.build_neighbours()
            s.eam_forces()
            s.step(4)
            _fresh[kind] = f0, s.positions(), s.forces()
    return _fresh[kind]


@pytest.mark.parametrize("kind,barrier", BARRIERS)
def test_timed_out_rebuild_recovers(kind, barrier):
    f0, pos, f1 = fresh(kind)
    # order of the FP64 half list's atomic adds; FP32 terms summed in the rows' order otherwise
    tol = 1e-11 if kind.startswith("fp64") else 1e-5
    with make(kind) as s:
        assert md.md_selftest_timeout_at(s.ctx, barrier) == md.MD_ERR_TIMEOUT
        s.eam_forces()
        assert np.abs(s.forces() - f0).max() <= tol * np.abs(f0).max()
        s.step(3)
        before = s.positions(), s.velocities()
        assert md.md_selftest_timeout_at(s.ctx, barrier) == md.MD_ERR_TIMEOUT
        assert np.array_equal(s.positions(), before[0]) and np.array_equal(s.velocities(), before[1])
        s.step(4)
        assert np.abs(s.positions() - pos).max() <= tol
        assert np.abs(s.forces() - f1).max() <= tol * np.abs(f1).max()


def test_contexts_without_a_barrier_say_so():
    w = I.fcc_cu(12, seed=3, n_knots=500)
    with md.System(w, precision="mixed", passes="staged") as s:
        assert md.md_selftest_timeout_at(s.ctx, 1) == 11   # wrong state
    with make("fp64-list") as s:
        assert md.md_selftest_timeout_at(s.ctx, 9) == md.md_selftest_timeout_at(s.ctx, 0) == 1   # bad argument


@pytest.mark.parametrize("kind", ["fp64-half", "mixed-list"])
def test_tuning_reports_a_trial_that_gave_up(kind):
    """A trial step that gives up would otherwise be the fastest of all."""
    f0, _, _ = fresh(kind)
    tol = 1e-11 if kind.startswith("fp64") else 1e-5
    with make(kind) as s:
        s.eam_forces()
        before = s.positions(), s.velocities()
        assert md.md_selftest_timeout_at(s.ctx, 11) == md.MD_ERR_TIMEOUT
        assert np.array_equal(s.positions(), before[0]) and np.array_equal(s.velocities(), before[1])
        s.eam_forces()
        assert np.abs(s.forces() - f0).max() <= tol * np.abs(f0).max()
        assert s.tune() in (1, 2, 4, 8, 16, 32)
        s.step(1)
