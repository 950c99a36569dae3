"""The steady solve on thread-block clusters (csrc/steady.cu) at the edges of
its splits: one and several CTAs per tissue, strips that do not fill, rows and
columns that do not divide, a solve longer than one launch, and lattices just
outside, which take the one-launch-per-step path."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lb():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1503_06726_gb300 import lbib
    return lbib


def relax(src, D, decay, rate, steps, phi0=None, check=16):
    """FP64 relaxation: phi after `steps` steps and the last check's residual."""
    w = np.array([1 / 3] + [1 / 6] * 4)
    move = [(0, 0), (0, 1), (1, 0), (0, -1), (-1, 0)]
    phi = np.zeros(src.shape) if phi0 is None else phi0
    g = w[:, None, None] * phi
    resid = np.inf
    pulled = lambda g: np.stack([np.roll(g[q], move[q], (0, 1)) for q in range(5)])
    for n in range(1, steps + 1):
        g = pulled(g)
        phi = g.sum(0)
        R = rate * src - decay * phi
        g = g + (w[:, None, None] * phi - g) / (3 * D + 0.5) + w[:, None, None] * R
        if n % check == 0:
            new = pulled(g).sum(0)
            resid = np.abs(new - phi).max() / np.abs(new).max()
    return pulled(g).sum(0), resid


# nx, ny, batch, steps: (8, 8) the smallest; 1024 wide is one strip per CTA;
# 1025 wide and 520 x 130 (more than 16 CTAs) do not fit in a cluster
SHAPES = [(8, 8, 1, 37), (97, 9, 3, 32), (31, 255, 5, 21), (256, 256, 2, 48), (300, 290, 1, 16),
          (1024, 12, 1, 17), (512, 64, 9, 15), (130, 66, 40, 33), (8, 9, 2, 8211),
          (1025, 16, 1, 33), (520, 130, 1, 16)]


@pytest.mark.parametrize("nx,ny,batch,steps", SHAPES)
@pytest.mark.parametrize("warm", [False, True])
def test_fixed_steps_match_fp64(lb, nx, ny, batch, steps, warm):
    import torch
    rng = np.random.default_rng(nx * 1000 + ny + batch)
    src = (rng.random((batch, ny, nx)) < 0.15).astype(np.uint8)
    src[:, 0, 0] = 1
    D, decay = rng.uniform(0.05, 0.2, batch), rng.uniform(1e-3, 1e-2, batch)
    rate = np.full(batch, 1e-3)
    # near the steady level, so that the watch keeps it
    phi0 = (0.15 * rate / decay)[:, None, None] * rng.uniform(0.9, 1.1, (batch, ny, nx)) \
        if warm else None
    t0 = None if phi0 is None else torch.as_tensor(phi0.astype(np.float32), device="cuda")
    phi, n, resid, fell = lb.steady_solve(torch.as_tensor(src, device="cuda"), D, decay, rate,
                                          phi0=t0, tol=0.0, max_steps=steps, with_fallback=True)
    # a residual of exactly zero (an FP32 fixed point) meets tol = 0 and ends early
    assert ((n == steps) | ((resid == 0.0) & (n < steps) & (n % 16 == 0))).all()
    phi = phi.cpu().numpy()
    for b in sorted({0, batch // 2, batch - 1}):
        if fell[b]:
            continue  # restarted from zero at a check of the watch
        want, r = relax(src[b], D[b], decay[b], rate[b], int(n[b]),
                        None if phi0 is None else phi0[b].astype(np.float32).astype(np.float64))
        # every step rounds phi and five populations once or twice (2^-24
        # each); the decay forgets errors older than 1 / decay steps
        bound = 8 * 2.0 ** -24 * min(steps, 2 / decay[b])
        assert np.abs(phi[b] - want).max() <= bound * np.abs(want).max()
        if steps >= 16:
            # the residual is a difference of two such fields
            assert abs(resid[b] - r) <= 2 * bound + 1e-3 * r
