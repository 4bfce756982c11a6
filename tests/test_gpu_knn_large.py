"""The grouped kNN kernel where its tree of boxes has a third triple of levels
(more than 8.4 million particles): lists, densities and r_k equal the
single-scan kernel's bit for bit, in one box whose particle count is no
multiple of a node and in subvolumes that start at odd offsets beyond it."""
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


def _clustered(n, seed):
    """60 % in clumps of about 3,000 whose sizes span two decades, the rest uniform."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    m, c = int(0.6 * n), max(1, n // 5000)
    which = torch.randint(c, (m,), generator=g, device="cuda")
    size = 10.0 ** (-2.0 - 2.0 * torch.rand(c, 1, generator=g, device="cuda"))
    centre = torch.rand(c, 3, generator=g, device="cuda")
    pos = torch.rand(n, 3, generator=g, device="cuda")
    pos[:m] = torch.remainder(centre[which] + size[which] * torch.randn(m, 3, generator=g, device="cuda"), 1.0)
    pos[pos >= 1.0] = 0.0
    return pos


def test_one_box(hop):
    pos = _clustered(9000011, 1)
    p = hopgpu.default_params(radius_mode=hopgpu.HOP_RADIUS_COUNT)
    out = []
    for tuning in ((4, 2, 0), (8, 1, 4)):
        hop.apply_tuning(*tuning)
        try:
            out.append(hop.hop_density(pos, p, ld_nbr=16, want_rk=True))
        finally:
            hop.apply_tuning(8, 1, 0)
    for x, y, name in zip(*out, ("nbr", "dens", "rk")):
        assert torch.equal(x, y), name


def test_subvolumes(hop):
    sizes = (8400011, 600001, 70001, 999)
    pos = torch.cat([_clustered(n, 10 + i) for i, n in enumerate(sizes)])
    off = [0]
    for n in sizes:
        off.append(off[-1] + n)
    p = hopgpu.default_params(radius_mode=hopgpu.HOP_RADIUS_COUNT)
    out = []
    for tuning in ((8, 2, 0), (8, 1, 4)):
        hop.apply_tuning(*tuning)
        try:
            out.append(hop.hop_run_batch(pos, off, [1.0] * len(sizes), p, ld_nbr=16))
        finally:
            hop.apply_tuning(8, 1, 0)
    for key in ("dens", "nbr", "group"):
        assert torch.equal(out[0][key], out[1][key]), key
