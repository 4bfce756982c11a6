"""The kernels that serve what the grouped kNN kernel hands over, on inputs
whose hand-over is certain: shells of more than Ndens + 32 particles around a
query, at one distance or so thin that the grouped kernel's bins (65,536 of
them in the limit) cannot divide them while the distances themselves can.  A
warp then lists the shell (up to 320 particles within the radius), counts again
in finer bins and scans a second time (more), or reports HOP_EDEGENERATE (more
than 320 at one distance).  Reference: the single-scan kernel, bit for bit, and
for the query in the middle the definition itself."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1001_3411_gb300 as hopgpu

pytestmark = pytest.mark.gpu
SCALE = 1024.0


@pytest.fixture(scope="module")
def hop():
    hopgpu.build_library()
    h = hopgpu.Hop(0)
    yield h
    h.close()


def _lattice_shell(least, most):
    """All integer offsets with one a^2 + b^2 + c^2 = S, for the smallest S
    with least .. most of them: their distances are equal in any precision."""
    r = np.arange(-48, 49)
    g = np.stack(np.meshgrid(r, r, r, indexing="ij"), -1).reshape(-1, 3)
    s = (g * g).sum(1)
    count = np.bincount(s)[: 48 * 48]
    S = int(np.flatnonzero((count >= least) & (count <= most))[0])
    return g[s == S], S


def _with_background(middle, shell, seed, n_bg=6000):
    """Middle, shell and a uniform background that stays out of the shell."""
    rng = np.random.default_rng(seed)
    bg = rng.random((4 * n_bg, 3))
    d = bg - middle
    d -= np.round(d)
    bg = bg[(d * d).sum(1) > 0.06 ** 2][:n_bg]
    return np.concatenate([shell, [middle], bg])


def _equal_shell(least, most):
    off, S = _lattice_shell(least, most)
    return _with_background(np.full(3, 0.5), 0.5 + off / SCALE, 3), len(off), S


def _thin_shell(n_shell, width, middle, seed=6):
    rng = np.random.default_rng(seed)
    v = rng.normal(size=(n_shell, 3))
    v /= np.linalg.norm(v, axis=1, keepdims=True)
    m = np.full(3, middle)
    return _with_background(m, m + 0.02 * v * (1 + width * rng.random((n_shell, 1))), 4)


def _density(hop, pos, tuning, ld=16, **kw):
    hop.apply_tuning(*tuning)
    try:
        return hop.hop_density(torch.from_numpy(pos).cuda(), hopgpu.default_params(**kw), ld_nbr=ld, want_rk=True)
    finally:
        hop.apply_tuning(8, 1, 0)


def _both(hop, pos, tuning, ld, **kw):
    a = _density(hop, pos, tuning, ld, **kw)
    b = _density(hop, pos, (8, 1, 4), ld, **kw)
    for x, y, name in zip(a, b, ("nbr", "dens", "rk")):
        assert torch.equal(x, y), name
    return a


@pytest.mark.parametrize("ld", [16, 64])
@pytest.mark.parametrize("qpw", [4, 8, 16])
def test_one_distance(hop, qpw, ld):
    """150 to 220 particles at the Ndens-th distance: within the 320 listed."""
    pos, m, S = _equal_shell(150, 220)
    nbr, _, rk = _both(hop, pos.astype(np.float32), (qpw, 2, 0), ld)
    assert nbr[m].tolist() == [m] + list(range(ld - 1))     # the middle, then the shell by index
    assert rk[m].item() == np.float32(np.sqrt(np.float32(S / SCALE ** 2)))


@pytest.mark.parametrize("f64", [False, True])
@pytest.mark.parametrize("qpw", [4, 8])
def test_more_at_one_distance_than_any_list_holds(hop, qpw, f64):
    pos, m, _ = _equal_shell(321, 100000)
    assert m > 320
    with pytest.raises(hopgpu.HopError) as err:
        _density(hop, pos.astype(np.float64 if f64 else np.float32), (qpw, 2, 0), pos_is_f64=int(f64))
    assert err.value.code == hopgpu.HOP_EDEGENERATE
    _both(hop, pos[m:].astype(np.float32), (qpw, 2, 0), 16)  # the context goes on


# float32: coordinates near 0.03 are 2e-9 apart, so the shell holds about 30
# distances, 20 particles at each.  Either way the shell is thinner than the
# 1.5e-5 that the grouped kernel's bins divide.
@pytest.mark.parametrize("ld", [16, 64])
@pytest.mark.parametrize("qpw", [4, 8, 16])
@pytest.mark.parametrize("n_shell", [250, 600])
def test_thin_shell(hop, n_shell, qpw, ld):
    _both(hop, _thin_shell(n_shell, 1e-6, 0.03).astype(np.float32), (qpw, 2, 0), ld)


@pytest.mark.parametrize("qpw", [1, 8, 32])
@pytest.mark.parametrize("n_shell", [250, 600])
def test_thin_shell_float64(hop, n_shell, qpw):
    _both(hop, _thin_shell(n_shell, 1e-9, 0.5), (qpw, 1, 0), 16, pos_is_f64=1)


@pytest.mark.parametrize("qpw", [4, 8])
def test_subvolumes(hop, qpw):
    parts = [_equal_shell(150, 220)[0].astype(np.float32), _thin_shell(600, 1e-6, 0.03).astype(np.float32),
             np.random.default_rng(9).random((65, 3)).astype(np.float32)]   # (too few for a ball that does not wrap)
    off = np.concatenate([[0], np.cumsum([len(x) for x in parts])])
    p = hopgpu.default_params()
    hop.apply_tuning(qpw, 2, 0)
    try:
        r = hop.hop_run_batch(torch.from_numpy(np.concatenate(parts)).cuda(), off, [1.0] * 3, p, ld_nbr=16)
    finally:
        hop.apply_tuning(8, 1, 0)
    for b, x in enumerate(parts):
        nbr, dens, _ = _density(hop, x, (8, 1, 4))
        assert torch.equal(r["dens"][off[b]:off[b + 1]], dens)
        assert torch.equal(r["nbr"][off[b]:off[b + 1]], nbr + int(off[b]))
