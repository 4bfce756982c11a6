"""The grouped kNN kernel (four queries per warp, eight lanes each) at the
sizes and shapes where it can go wrong: counts around its groups and nodes,
boxes so small that queries are handed over to the warp-per-query kernel,
balls across faces, the shortest and longest lists, particles far from their
neighbours in the sort order.  Reference: the single-scan kernel, whose results are
exact too, so lists, densities and r_k must be equal bit for bit."""
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


def _both(hop, pos, qpw=4, cpr=2, ld=16, **kw):
    p = hopgpu.default_params(**kw)
    pos = torch.from_numpy(np.ascontiguousarray(pos)).cuda()
    out = []
    for tuning in ((qpw, cpr, 0), (8, 1, 4)):
        hop.apply_tuning(*tuning)
        try:
            out.append(hop.hop_density(pos, p, ld_nbr=ld, want_rk=True))
        finally:
            hop.apply_tuning(8, 1, 0)
    for x, y, name in zip(*out, ("nbr", "dens", "rk")):
        assert torch.equal(x, y), name


@pytest.mark.parametrize("n", [64, 65, 127, 129, 511, 513, 1021, 4095, 4097, 32771, 50021, 100003])
@pytest.mark.parametrize("qpw", [4, 16])
def test_counts_around_groups_and_nodes(hop, n, qpw):
    _both(hop, synth.uniform_box(n, 300 + n), qpw=qpw)


@pytest.mark.parametrize("k,ld,n_hop", [(2, 2, 1), (3, 3, 3), (32, 8, 8), (65, 65, 65), (128, 128, 128), (128, 16, 4)])
def test_list_lengths(hop, k, ld, n_hop):
    _both(hop, synth.nfw_box(20003, 21)[0], ld=ld, n_dens=k, n_hop=n_hop, n_merge=1)


@pytest.mark.parametrize("box", [1e-3, 0.37, 250.0])
@pytest.mark.parametrize("mode", [0, 1])
def test_boxes_and_faces(hop, box, mode):
    """Clumps on the faces, edges and corners of the box."""
    rng = np.random.default_rng(3)
    c = np.array([[0, 0, 0], [0, 0.5, 0.5], [0.5, 0, 0], [0.25, 0.75, 0]])
    pos = np.concatenate([c[rng.integers(0, 4, 9000)] + 0.03 * rng.normal(size=(9000, 3)), rng.random((3001, 3))])
    pos = synth._wrap_f32(pos * box, box)
    _both(hop, pos, box=box, radius_mode=mode)


@pytest.mark.parametrize("cpr", [1, 3])
def test_sparse_and_dense_neighbours(hop, cpr):
    """Tight pairs of clumps in an almost empty box: first radii far too
    large and far too small, jumps of the sort order inside a group."""
    rng = np.random.default_rng(8)
    cen = rng.random((40, 3))
    size = rng.integers(1, 400, 40)
    pos = np.concatenate([c + 10.0 ** -rng.uniform(1.5, 5) * rng.normal(size=(s, 3)) for c, s in zip(cen, size)])
    pos = synth._wrap_f32(np.concatenate([pos, rng.random((100, 3))]) % 1.0, 1.0)
    for mode in (0, 1):
        _both(hop, pos, cpr=cpr, radius_mode=mode)


@pytest.mark.parametrize("qpw", [4, 8, 16])
@pytest.mark.parametrize("sizes", [(65, 999, 64, 5001), (30011, 513, 70001, 8191)])
def test_subvolumes_at_odd_offsets(hop, sizes, qpw):
    """Runs of eight particles that straddle two subvolumes."""
    boxes = [1.0, 0.25, 3.0, 1.0]
    pos = np.concatenate([synth._wrap_f32(synth.nfw_box(n, 70 + i)[0].astype(np.float64) * b, b)
                          for i, (n, b) in enumerate(zip(sizes, boxes))])
    off = np.concatenate([[0], np.cumsum(sizes)])
    pos = torch.from_numpy(pos).cuda()
    out = []
    for tuning in ((qpw, 2, 0), (8, 1, 4)):
        hop.apply_tuning(*tuning)
        try:
            out.append(hop.hop_run_batch(pos, off, boxes, hopgpu.default_params(), ld_nbr=16))
        finally:
            hop.apply_tuning(8, 1, 0)
    for key in ("dens", "nbr", "group"):
        assert torch.equal(out[0][key], out[1][key]), key


F64_CASES = {
    "plummer": lambda: synth.workload("plummer32k"),
    "lattice": lambda: synth.lattice_box(16, dtype=np.float64),
    "uniform": lambda: synth.uniform_box(20011, 5, dtype=np.float64),
    "tiny": lambda: synth.uniform_box(130, 6, dtype=np.float64),
    # distances far below a float's spacing at the coordinates' size
    "tight": lambda: np.concatenate([0.7 + 1e-7 * np.random.default_rng(4).random((300, 3)),
                                     np.random.default_rng(5).random((3000, 3))]),
}


@pytest.mark.parametrize("qpw", [1, 8, 32])
@pytest.mark.parametrize("case", list(F64_CASES))
def test_float64(hop, case, qpw):
    _both(hop, F64_CASES[case](), qpw=qpw, pos_is_f64=1)


@pytest.mark.parametrize("box", [1e-3, 250.0])
def test_float64_boxes_and_lists(hop, box):
    pos = (synth.nfw_box(20001, 31, dtype=np.float64)[0] * box) % box
    for k, ld, mode in ((64, 64, 0), (65, 65, 1), (128, 16, 1), (2, 2, 0)):
        _both(hop, pos, box=box, ld=ld, n_dens=k, n_hop=min(ld, k), n_merge=1, radius_mode=mode, pos_is_f64=1)
