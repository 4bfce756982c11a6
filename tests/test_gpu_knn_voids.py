"""Particles in a void around a ball of more 512-particle nodes than the
grouped kNN kernel lists, with the plain first radius: the group's region meets
the whole ball long before a query's own does.  Lists, densities and r_k must
equal the single-scan kernel's bit for bit, and no query may be searched again
and again: between the first radius (0.05 of the box) and the largest served
(0.25) a radius that held too few grows by at least 1.25, which is at most
eight searches per particle in the void."""
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


def _directions(rng, n):
    v = rng.normal(size=(n, 3))
    return v / np.linalg.norm(v, axis=1, keepdims=True)


@pytest.mark.parametrize("n_ball,size,lo,hi", [(61440, 0.02, 0.12, 0.16), (100000, 0.02, 0.08, 0.1),
                                               (150000, 0.01, 0.08, 0.1)])
def test_voids_beside_a_ball(hop, n_ball, size, lo, hi):
    rng = np.random.default_rng(5)
    n_void = 200
    pos = np.concatenate([0.5 + _directions(rng, n_ball) * size * rng.random((n_ball, 1)) ** (1 / 3),
                          0.5 + _directions(rng, n_void) * rng.uniform(lo, hi, (n_void, 1))])
    pos = torch.from_numpy(pos.astype(np.float32)).cuda()
    p = hopgpu.default_params()
    out, retries = [], []
    for tuning in ((8, 1, 0), (8, 1, 4)):
        hop.apply_tuning(*tuning)
        try:
            out.append(hop.hop_density(pos, p, ld_nbr=16, want_rk=True))
            retries.append(hop.stats()["retries"])
        finally:
            hop.apply_tuning(8, 1, 0)
    for x, y, name in zip(*out, ("nbr", "dens", "rk")):
        assert torch.equal(x, y), name
    assert retries[0] <= 8 * n_void
