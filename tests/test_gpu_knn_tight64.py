"""Float64 particles packed closer than float32 tells apart at their
coordinates: whole nodes of the sorted particles go to the kernel that works in
double, four consecutive queries per warp, and radii that float32 cannot bin
are given up at once.  Reference: the single-scan kernel over every query;
lists, densities and r_k must be equal bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1001_3411_gb300 as hopgpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hop():
    hopgpu.build_library()
    h = hopgpu.Hop(0)
    yield h
    h.close()


def _ball(rng, n, centre, size):
    v = rng.normal(size=(n, 3))
    v *= size * rng.random((n, 1)) ** (1 / 3) / np.linalg.norm(v, axis=1, keepdims=True)
    return np.asarray(centre) + v


def _points(case, rng):
    if case == "one":           # 117 tight nodes, more than the kernel lists
        return [_ball(rng, 60000, (0.5, 0.5, 0.5), 1e-6), rng.random((3000, 3))]
    if case == "edges":         # sizes around one and two nodes, on both sides of the limit, across a face
        return [_ball(rng, 511, (0.2, 0.3, 0.4), 1e-7), _ball(rng, 513, (0.7, 0.3, 0.4), 1e-9),
                _ball(rng, 1025, (0.0, 0.5, 1.0), 1e-7), _ball(rng, 2000, (0.1, 0.8, 0.8), 4e-6),
                _ball(rng, 2000, (0.6, 0.8, 0.8), 1e-5), rng.random((3001, 3))]
    return [_ball(rng, 700, c, 2e-7) for c in rng.random((40, 3))]   # tight nodes and nodes of two balls


@pytest.mark.parametrize("qpw", [1, 4, 8])
@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("case", ["one", "edges", "many"])
def test_tight_float64(hop, case, mode, qpw):
    pos = np.concatenate(_points(case, np.random.default_rng(23))) % 1.0
    dev = torch.from_numpy(pos).cuda()
    p = hopgpu.default_params(pos_is_f64=1, radius_mode=mode)
    out, stats = [], []
    for tuning in ((qpw, 1, 0), (8, 1, 4)):
        hop.apply_tuning(*tuning)
        try:
            out.append(hop.hop_density(dev, p, ld_nbr=16, want_rk=True))
            stats.append(hop.stats())
        finally:
            hop.apply_tuning(8, 1, 0)
    for x, y, name in zip(*out, ("nbr", "dens", "rk")):
        assert torch.equal(x, y), name
    if case == "one":
        # first tries: one per four particles of the ball, and at most two per
        # particle outside or in a node with some outside (two of them in each
        # of the eight octants that meet in the ball), not one per particle
        assert stats[0]["searches"] - stats[0]["retries"] <= 60000 // 4 + 2 * (3000 + 16 * 512)
