"""One-species tables at FP64, whose pair terms are built from FP32 pieces and whole numbers: coarse
and fine tables, knots off the binary fractions, pairs below the first knot, and tables outside the
pieces' range (more than 20,000 knots, a first knot near 0), which keep FP64 arithmetic; the item
walks (1 and 2 lanes an atom) and the flattened ones, full and half lists, a cubic and an uneven box
with atoms on its faces.  Forces, energy, rho and virial against the oracle at the FP64 bar of 1e-10."""
import dataclasses

import numpy as np
import pytest

import oracle
from paper_1107_2619_gb300 import inputs as I, md

pytestmark = pytest.mark.gpu

TOL = 1e-10


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1107_2619_gb300 import build
    build.build()


def crystal(n_knots, r_min, uneven):
    w = I.fcc_cu(8, seed=n_knots, sigma=0.08)
    pos, box = w.pos.copy(), w.box.copy()
    if uneven:   # a stretched box, shifted so that planes of atoms straddle its faces
        scale = np.array([1.0, 1.013, 0.994])
        box = box * scale
        pos = np.mod(pos * scale + np.array([0.0, 0.02, -0.03]), box)
        pos[np.argmin(pos[:, 0]), 0] = 0.0
        pos[np.argmax(pos[:, 1]), 1] = np.nextafter(box[1], 0.0)
    return dataclasses.replace(w, pos=pos, box=box, potential=I.sc_cu_tables(n_knots=n_knots, r_min=r_min))


@pytest.mark.parametrize("walk,lanes", [("auto", 1), ("auto", 8), ("half", 2), ("half", 4), ("half", 16)])
@pytest.mark.parametrize("n_knots,r_min,uneven", [
    (5000, 1.0, False), (60, 1.3, True), (777, 1.7, True), (20000, 0.9, False), (5000, 2.45, True),
    (20001, 1.0, False), (5000, 0.05, True)])
def test_table_pairs_match_oracle(n_knots, r_min, uneven, walk, lanes):
    w = crystal(n_knots, r_min, uneven)
    ref = oracle.forces(w.pos, w.species, w.box, w.potential, skin=w.skin, k_max=w.k_max, method="brute")
    with md.System(w, precision="fp64", passes=walk, lanes_per_atom=lanes) as s:
        pe = s.eam_forces()
        f, e, rho = s.forces(), s.energy(), s.get(md.MD_GET_RHO)
    assert np.abs(f - ref["force"]).max() <= TOL * np.abs(ref["force"]).max()
    assert abs(pe - ref["pe"]) <= TOL * abs(ref["pe"])
    assert np.abs(rho - ref["rho"]).max() <= TOL * np.abs(ref["rho"]).max()
    assert np.abs(e["virial"] - ref["virial"]).max() <= TOL * np.abs(ref["virial"]).max()
