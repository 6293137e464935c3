"""The list walk's per-atom work by whole warps, and the placement of a moved atom: sizes whose last
batch is partial at every lane count, and atoms far outside the box (their image taken off from
the build's record: by small whole numbers, and beyond what the record holds).  Against the
oracle's velocity Verlet, with the bounds of the other trajectory tests (FP64: 1e-9 Å plus the
rounding of the coordinates themselves; mixed: 1e-4 Å)."""
import dataclasses

import numpy as np
import pytest

import oracle
from paper_1107_2619_gb300 import inputs as I, md

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1107_2619_gb300 import build
    build.build()


@pytest.mark.parametrize("lanes", [1, 2, 8, 32])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("shift", [(0, 0, 0), (3, -2, 0), (700, 0, -511)])
def test_partial_batches_and_far_images_match_oracle(lanes, precision, shift):
    w = I.bcc_fe(0, seed=21, temperature=900.0, cells=(5, 6, 7))   # 420 atoms
    assert w.n_atoms % 32 != 0
    # every third atom sits whole boxes away
    far = np.arange(w.n_atoms) % 3 == 1
    w = dataclasses.replace(w, pos=w.pos + far[:, None] * np.array(shift) * w.box)
    steps = 40
    with md.System(w, precision=precision, lanes_per_atom=lanes) as s:
        s.step(steps)
        pos, e = s.positions(), s.energy()
    assert e["n_rebuilds"] >= 3
    ref = oracle.run_vv(w.pos, w.vel, w.species, w.potential.masses, w.box, w.potential, w.dt_fs, steps, w.skin, w.k_max)
    ulp = np.spacing(np.abs(w.pos).max())
    tol = 1e-9 + 2 * steps * ulp if precision == "fp64" else 1e-4
    assert np.abs(pos - ref["pos"]).max() < tol
