"""The lattice fields of lbib_get_fields at the sizes where their way to the
host changes, against the oracle: the last lattice converted on the host, the
first packed on the device, one that needs several trips through the staging
region (16 MB: 2 M doubles), rows longer than the region's chunk is high, and
fields asked for one at a time."""
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


# 65,535 nodes, 65,536 nodes, 2.2 M nodes, and 70,000 columns in 32 rows
@pytest.mark.parametrize("nx,ny", [(257, 255), (256, 256), (1531, 1437), (70000, 32)])
@pytest.mark.parametrize("precision", ["fp32", "fp64", "fp16"])
def test_fields_match_oracle(lb, orc, nx, ny, precision):
    rng = np.random.Generator(np.random.PCG64(3))
    P = li.LatticeParams(nx=nx, ny=ny, bc_y=li.BC_PERIODIC, tau=0.8, n_species=2)
    for s in range(2):
        P.D[s], P.decay[s], P.src_rate[s] = 0.1, 1e-3, 1e-3 * (s + 1)
    centres = [(nx * 0.3, ny * 0.5), (nx * 0.9, ny * 0.4)]
    T = li.make_tissue(centres, np.full(2, 9.0), 40, 0.01, 1e-3,
                       np.array([1, 2], np.uint8), jitter=0.2, rng=rng)
    n = 4
    sim = lb.Simulation(P, lb.PRECISIONS[precision], T.n_vertices, T.n_cells)
    sim.set_cells(T)
    sim.step(n)
    bits = [lb.LBIB_RHO, lb.LBIB_U, lb.LBIB_PHI, lb.LBIB_ID, lb.LBIB_FORCE]
    got = sim.fields(sum(bits) | lb.LBIB_X)
    for b in bits:  # the same alone
        for key, v in sim.fields(b).items():
            assert np.array_equal(v, got[key]), key
    sim.close()
    ref = orc.run(P, T, n)
    assert np.array_equal(got["id"], ref.id)
    rel = lambda a, b: float(np.abs(a - b).max() / max(np.abs(b).max(), 1e-300))
    # the bounds of the FP64, FP32 (1e-10; u 1e-4, phi 1e-5) and FP16 paths
    # (phi 1e-2; rho to its storage step, u and the force not compared)
    br, bu, bp = {"fp64": (1e-10, 1e-10, 1e-10), "fp32": (1e-5, 1e-4, 1e-5),
                  "fp16": (1e-3, None, 1e-2)}[precision]
    assert rel(got["rho"], ref.rho) < br
    assert rel(got["phi"], ref.phi) < bp
    if bu is not None:
        assert max(rel(got["ux"], ref.ux), rel(got["uy"], ref.uy)) < bu
        assert rel(got["force"], np.stack([ref.fx, ref.fy], axis=-1)) < bu
