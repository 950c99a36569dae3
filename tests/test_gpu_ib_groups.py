"""The immersed-boundary work at the edges of its per-cell table of force groups
(csrc/ib_cell.cuh, GroupBox) and of its row accesses, against the oracle: a
cell across the periodic seams, cells just inside and outside the table's
64-node width, stencils at walls, even and odd columns, more vertices than
threads, and enough cells for the small-CTA kernels."""
import numpy as np
import pytest

import lbib_inputs as li

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1503_06726_gb300 import build, lbib
    build.build()
    lbib.load()
    return lbib


def workload(nx, ny, centres, radius, n_vert, walls=False, seed=5):
    rng = np.random.Generator(np.random.PCG64(seed))
    P = li.LatticeParams(nx=nx, ny=ny, bc_y=li.BC_WALLS if walls else li.BC_PERIODIC, tau=0.8,
                         n_species=1)
    P.D[0], P.decay[0], P.src_rate[0] = 0.1, 1e-3, 1e-3
    src = (np.arange(len(centres)) % 2 == 0).astype(np.uint8)
    T = li.make_tissue(centres, np.full(len(centres), radius), n_vert, 0.01, 1e-3, src,
                       jitter=0.2, rng=rng)
    return P, T


CASES = {
    # across both seams, and a cell of the same shape away from them
    "seams": (96, 80, [(1.0, 2.0), (50.0, 40.0)], 12.0, 48, False),
    # stencil boxes of 62 .. 66 nodes: inside, at and outside 16 groups
    "width_62": (128, 100, [(64.25, 50.0)], 29.1, 90, False),
    "width_64": (128, 100, [(63.5, 50.0)], 30.2, 90, False),
    "width_66": (128, 100, [(64.0, 50.0)], 31.3, 90, False),
    # higher than the table's 128 rows, more vertices than the CTA's threads
    "high": (200, 190, [(100.0, 95.0)], 70.0, 300, False),
    # the stencils reach the wall rows
    "walls": (97, 65, [(30.0, 13.5), (66.0, 50.6)], 12.0, 40, True),
    # one row of nodes per vertex shift: odd lattice width, triangles
    "triangles": (33, 31, [(9.0, 9.0), (24.0, 22.0)], 5.0, 3, False),
}


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_cells_match_oracle(lb, orc, name, precision):
    nx, ny, centres, radius, n_vert, walls = CASES[name]
    P, T = workload(nx, ny, centres, radius, n_vert, walls)
    n = 20
    sim = lb.Simulation(P, lb.PRECISIONS[precision], T.n_vertices, T.n_cells)
    sim.set_cells(T)
    sim.step(n)
    got = sim.fields(lb.LBIB_U | lb.LBIB_PHI | lb.LBIB_X | lb.LBIB_ID | lb.LBIB_FORCE)
    ref = orc.run(P, T, n)
    assert np.array_equal(got["id"], ref.id)
    rel = lambda a, b: float(np.abs(a - b).max() / max(np.abs(b).max(), 1e-300))
    # the bounds of the FP64 and FP32 paths (1e-10; u 1e-4, phi 1e-5, X 1e-6)
    bu, bp, bx = (1e-10, 1e-10, 1e-10) if precision == "fp64" else (1e-4, 1e-5, 1e-6)
    assert max(rel(got["ux"], ref.ux), rel(got["uy"], ref.uy)) < bu
    assert rel(got["phi"], ref.phi) < bp
    assert np.abs(got["xy"] - ref.xy).max() < bx
    f = np.stack([ref.fx, ref.fy], axis=-1)
    assert rel(got["force"], f) < bu
    sim.close()


@pytest.mark.parametrize("n_vert", [64, 100])
def test_many_small_cells_match_oracle(lb, orc, n_vert):
    """2,116 cells: the 64- and 128-thread kernels."""
    side, pitch = 46, 14.0
    n = int(side * pitch)
    centres = [(pitch * (i + 0.5) + 0.37 * j % 1.0, pitch * (j + 0.5)) for j in range(side)
               for i in range(side)]
    P, T = workload(n, n, centres, 5.0, n_vert)
    sim = lb.Simulation(P, lb.LBIB_FP32, T.n_vertices, T.n_cells)
    sim.set_cells(T)
    sim.step(5)
    got = sim.fields(lb.LBIB_U | lb.LBIB_X | lb.LBIB_ID)
    ref = orc.run(P, T, 5)
    assert np.array_equal(got["id"], ref.id)
    rel = lambda a, b: float(np.abs(a - b).max() / max(np.abs(b).max(), 1e-300))
    assert max(rel(got["ux"], ref.ux), rel(got["uy"], ref.uy)) < 1e-4
    assert np.abs(got["xy"] - ref.xy).max() < 1e-6
    sim.close()
