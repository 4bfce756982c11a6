"""Box sides far from 1 (a catalogue in metres has 1e22 and more per
megaparsec): the float32 squares of such coordinates leave float32's range, so
float64 particles are searched in units of the box and float32 ones beyond
2^-50 .. 2^60 by the warp-per-query kernel.  A power of two scales positions
exactly, so lists and densities must equal those of the unit box bit for bit;
other sides are compared with the single-scan kernel, which works in double."""
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


def _density(hop, pos, tuning=(8, 1, 0), ld=16, **kw):
    hop.apply_tuning(*tuning)
    try:
        return hop.hop_density(torch.from_numpy(pos).cuda(), hopgpu.default_params(**kw), ld_nbr=ld, want_rk=True)
    finally:
        hop.apply_tuning(8, 1, 0)


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("n", [20000, 60000])
@pytest.mark.parametrize("box", [1e-25, 1e-20, 3e22, 3e24])
def test_float64_equals_single_scan(hop, box, n, mode):
    pos = (synth.nfw_box(n, 41, dtype=np.float64)[0] * box) % box
    a = _density(hop, pos, box=box, pos_is_f64=1, radius_mode=mode)
    b = _density(hop, pos, (8, 1, 4), box=box, pos_is_f64=1, radius_mode=mode)
    for x, y, name in zip(a, b, ("nbr", "dens", "rk")):
        assert torch.equal(x, y), name


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("e", [-330, -140, -67, 67, 79, 140, 330])
def test_float64_scaled_by_a_power_of_two(hop, e, mode):
    pos = synth.nfw_box(20011, 42, dtype=np.float64)[0]
    a = _density(hop, np.ldexp(pos, e), box=2.0 ** e, pos_is_f64=1, radius_mode=mode)
    b = _density(hop, pos, pos_is_f64=1)
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
    if abs(e) < 120:     # r_k is returned in float32
        assert np.array_equal(np.ldexp(a[2].cpu().numpy().astype(np.float64), -e), b[2].cpu().numpy())


def _grid_points(n, seed):
    """Coordinates on multiples of 1/1024: no square of a difference is a
    float32 denormal at any of the sides below."""
    return (np.random.default_rng(seed).integers(0, 1024, (n, 3)) / 1024.0).astype(np.float32)


# float32 densities are not compared: L^3 itself leaves float32's range
@pytest.mark.parametrize("e", [-51, -50, -49, 59, 60, 61])
def test_float32_scaled_by_a_power_of_two(hop, e):
    pos = _grid_points(20011, 43)
    a = _density(hop, np.ldexp(pos, e), box=2.0 ** e)
    b = _density(hop, pos)
    assert torch.equal(a[0], b[0])
    assert np.array_equal(np.ldexp(a[2].cpu().numpy().astype(np.float64), -e), b[2].cpu().numpy())


def test_float32_subvolumes_of_any_side(hop):
    sizes, exps = (5000, 3001, 777, 4096), (0, 61, -51, 2)
    parts = [_grid_points(n, 50 + i) for i, n in enumerate(sizes)]
    off = np.concatenate([[0], np.cumsum(sizes)])
    p = hopgpu.default_params()
    a = hop.hop_run_batch(torch.from_numpy(np.concatenate([np.ldexp(x, e) for x, e in zip(parts, exps)])).cuda(), off,
                          [2.0 ** e for e in exps], p, ld_nbr=16)
    b = hop.hop_run_batch(torch.from_numpy(np.concatenate(parts)).cuda(), off, [1.0] * 4, p, ld_nbr=16)
    assert torch.equal(a["nbr"], b["nbr"])


def test_float32_distances_beyond_float32_are_refused(hop):
    pos = _grid_points(20000, 44)
    with pytest.raises(hopgpu.HopError) as err:
        _density(hop, pos * np.float32(1e21), box=1e21)
    assert err.value.code == hopgpu.HOP_ETIMEOUT
    # the context goes on, and the same particles in float64 are served
    a = _density(hop, np.ldexp(pos.astype(np.float64), 70), box=2.0 ** 70, pos_is_f64=1)
    b = _density(hop, pos.astype(np.float64), pos_is_f64=1)
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
