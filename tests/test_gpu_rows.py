"""List rows and gathers at the edges of their 32-wide walks: cells from empty to more than 32
atoms and systems from fewer cells than warps to more (slices), row lengths around multiples of
32, and rows of more than 32 pairs in the surrogate's gathers.  The lists against the oracle's
sets, the surrogate's forces within the stated FP32 bound of the other surrogate tests (1e-4 of
the largest force)."""
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


@pytest.mark.parametrize("walk", ["auto", "half"])
@pytest.mark.parametrize("cells,kind", [(3, "random"), (4, "edges"), (9, "sparse")])
def test_rows_of_uneven_cells_match_oracle(walk, cells, kind):
    rng = np.random.default_rng(cells)
    n = cells ** 3
    if kind == "random":
        counts = rng.integers(0, 12, n)
    elif kind == "edges":   # one home more and less than a round of lanes, and empty cells
        counts = np.resize([0, 1, 31, 0, 33, 2, 0, 5], n)
    else:
        counts = (rng.random(n) < 0.2).astype(int)
    w = I.cell_count_gas(counts, cells=cells, seed=cells, k_max=256)
    with md.System(w, precision="fp64", passes=walk) as s:
        s.build_neighbours()
        cnt, lst = s.neighbours()
    count, rows, longest = oracle.neighbours(w.pos, w.box, w.potential.r_cut + w.skin, w.k_max)
    assert longest <= w.k_max and np.array_equal(cnt, count)
    for i in range(w.n_atoms):
        assert set(lst[i, :cnt[i]]) == set(rows[i, :cnt[i]]), i


@pytest.mark.parametrize("a,pairs", [(2.40, (33, 60)), (2.8665, (14, 27)), (3.7, (1, 20))])
def test_surrogate_rows_shorter_and_longer_than_a_warp(a, pairs):
    spec = dict(I.SUR_FE, k_max=96)
    cells = max(6, int(np.ceil(3.05 * 4.3 / a)))
    w = I.bcc_fe(0, seed=5, temperature=300.0, sigma=0.04, a=a, cells=(cells, cells, cells + 1))
    th = I.sur_init_weights(3, spec).astype(np.float32)
    with md.SurrogateSystem(w, th, net="fp32", spec=spec) as s:
        s.eam_forces()
        F, G, e = s.forces(), s.descriptors(), s.energy()
    o = oracle.surrogate(w.pos, w.box, spec, th.astype(np.float64), k_max=96)
    near = np.sqrt(((w.pos - w.pos[0] - w.box * np.rint((w.pos - w.pos[0]) / w.box)) ** 2).sum(1))
    assert pairs[0] <= int(((near > 0) & (near < spec["rd"])).sum()) <= pairs[1]
    assert np.abs(G - o["G"]).max() <= 2e-5 * max(1.0, np.abs(o["G"]).max())
    assert np.abs(F - o["force"]).max() <= 1e-4 * np.abs(o["force"]).max()
    assert abs(e["pe"] - o["energy"]) <= 2e-5 * max(1.0, np.abs(o["e_atom"]).max()) * w.n_atoms
