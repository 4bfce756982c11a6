"""Crowded lists of the grouped kNN kernel: a query's lists fill up while its
Ndens-th distance lies in the innermost or the outermost part of its first
radius, or its ball meets more boxes than the kernel lists.  Reference: the
single-scan kernel, whose results are exact too, so lists, densities and r_k
must be equal bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1001_3411_gb300 as hopgpu
import synth

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


def _points(shape):
    rng = np.random.default_rng(17)
    if shape == "cusp":            # radii over five decades
        return 0.5 + _directions(rng, 20000) * 10.0 ** -rng.uniform(0.8, 6, (20000, 1))
    if shape.startswith("shell"):  # a few particles inside thin shells
        width = float(shape[6:])
        c = np.array([[0.3, 0.3, 0.3], [0.7, 0.6, 0.4], [0.02, 0.5, 0.98]])
        shells = [x + _directions(rng, 3000) * 0.08 * (1 + width * rng.random((3000, 1))) for x in c]
        return np.concatenate(shells + [x + 1e-3 * rng.normal(size=(9, 3)) for x in c])
    # "outliers": a dense ball of 120 nodes, loners whose balls hold all of it
    ball = 0.5 + _directions(rng, 61440) * 0.04 * rng.random((61440, 1)) ** (1 / 3)
    return np.concatenate([ball, 0.5 + _directions(rng, 50) * rng.uniform(0.12, 0.2, (50, 1))])


@pytest.mark.parametrize("f64", [False, True])
@pytest.mark.parametrize("k", [3, 64, 128])
@pytest.mark.parametrize("shape", ["cusp", "shell 0.1", "shell 1e-3", "shell 1e-6", "outliers"])
def test_crowds(hop, shape, k, f64):
    pos = _points(shape) % 1.0
    pos = torch.from_numpy(pos if f64 else synth._wrap_f32(pos, 1.0)).cuda()
    p = hopgpu.default_params(n_dens=k, n_hop=3, n_merge=3, pos_is_f64=int(f64))
    out = []
    for tuning in ((8, 1, 0), (8, 1, 4)):
        hop.apply_tuning(*tuning)
        try:
            out.append(hop.hop_density(pos, p, ld_nbr=3, want_rk=True))
        finally:
            hop.apply_tuning(8, 1, 0)
    for x, y, name in zip(*out, ("nbr", "dens", "rk")):
        assert torch.equal(x, y), name
