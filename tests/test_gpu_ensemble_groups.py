"""Large ensembles, whose tissues form two groups on two streams, against the
same tissues run one by one: below and above the 500,000 nodes at which the
groups begin, calls shorter and longer than the 16 steps that the groups take
in turn, a last tissue larger than all others (a single group), and a group
without cells.

Tolerances as in the tests of small ensembles (the same kernels, only the
atomic order of the spreading differs: relative 1e-5 on u and phi, 1e-9 LU on
the vertices over ten steps; 1e-8 LU over the 40 here)."""
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


def tissue(nx, ny, cells, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    P = li.LatticeParams(nx=nx, ny=ny, bc_y=li.BC_PERIODIC, tau=0.8 + 0.01 * seed, n_species=1)
    P.D[0], P.decay[0], P.src_rate[0] = 0.1, 1e-3, 1e-3
    centres = [(nx * (i + 0.5) / max(cells, 1), ny * 0.5) for i in range(cells)]
    T = li.make_tissue(centres, np.full(cells, 9.0), 40, 0.01, 1e-3,
                       np.ones(cells, np.uint8), jitter=0.2, rng=rng) if cells else None
    return P, T


SIZES = {
    "one_group": [(96, 64, 2), (300, 200, 3)],
    "two_groups": [(512, 300, 4), (97, 65, 1), (640, 500, 3), (400, 333, 2)],
    "largest_last": [(96, 80, 1), (130, 100, 2), (900, 700, 4)],
    "no_cells_first": [(600, 500, 0), (512, 600, 3)],
}


@pytest.mark.parametrize("name", sorted(SIZES))
def test_groups_match_single_tissues(lb, name):
    every = [tissue(nx, ny, c, k + 1) for k, (nx, ny, c) in enumerate(SIZES[name])]
    ens = lb.Ensemble([p for p, _ in every], [t for _, t in every])
    assert ens.schedule() == lb.LBIB_ENS_SPLIT_WIDE
    calls = (1, 5, 34)
    for n in calls:
        ens.step(n)
    ens.status()
    for k, (P, T) in enumerate(every):
        nv, nc = (T.n_vertices, T.n_cells) if T is not None else (0, 0)
        sim = lb.Simulation(P, lb.LBIB_FP32, nv, nc)
        if T is not None:
            sim.set_cells(T)
        for n in calls:
            sim.step(n)
        a, b = ens.fields(k), sim.fields()
        sim.close()
        assert max(np.abs(a["ux"] - b["ux"]).max(), np.abs(a["uy"] - b["uy"]).max()) <= \
            1e-5 * max(np.abs(b["ux"]).max(), np.abs(b["uy"]).max()), k
        assert np.abs(a["phi"] - b["phi"]).max() <= 1e-5 * np.abs(b["phi"]).max(), k
        if T is not None:
            assert np.abs(a["xy"] - b["xy"]).max() < 1e-8, k
    ens.close()
