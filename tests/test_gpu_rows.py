"""Reading and writing neighbour rows in 16-byte parts: hops from rows of
every length and alignment against numpy, and lists written to rows of every
length (whole parts or single entries) against each other."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1001_3411_gb300 as hopgpu
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def case():
    hopgpu.build_library()
    h = hopgpu.Hop(0)
    pos = torch.from_numpy(synth.nfw_box(30011, 5)[0]).cuda()
    nbr, dens, _ = h.hop_density(pos, hopgpu.default_params(), ld_nbr=64)
    yield h, pos, nbr, dens
    h.close()


@pytest.mark.parametrize("offset", [0, 1, 2])
@pytest.mark.parametrize("ld,n_hop", [(1, 1), (3, 2), (4, 4), (8, 3), (8, 8), (16, 16), (17, 16), (20, 12), (64, 64)])
def test_hops_from_rows_of_every_shape(case, ld, n_hop, offset):
    h, _, nbr, dens = case
    n = len(dens)
    flat = torch.empty(n * ld + offset, dtype=torch.int32, device="cuda")
    rows = flat[offset:].view(n, ld)
    rows.copy_(nbr[:, :ld])
    hop, chain = h.hop_link(dens, rows, n_hop)
    d, r = dens.cpu().numpy().astype(np.float64), rows[:, :n_hop].cpu().numpy()
    key = np.lexsort((np.arange(n), -d))          # densest first, then the smaller index
    rank = np.empty(n, dtype=np.int64)
    rank[key] = np.arange(n)
    best = r[np.arange(n), np.argmin(rank[r], axis=1)]
    assert np.array_equal(hop.cpu().numpy(), best)
    top = best.copy()
    while not np.array_equal(top, best[top]):
        top = best[top]
    assert np.array_equal(chain.cpu().numpy(), top)


@pytest.mark.parametrize("ld", [16, 17, 18, 20, 63])
def test_rows_of_every_length_are_written_whole(case, ld):
    h, pos, nbr, dens = case
    a, d, _ = h.hop_density(pos, hopgpu.default_params(), ld_nbr=ld)
    assert torch.equal(a, nbr[:, :ld]) and torch.equal(d, dens)


def test_a_bad_index_in_a_row_is_reported(case):
    h, _, nbr, dens = case
    rows = nbr[:, :16].contiguous()
    for col, value in ((0, len(dens)), (5, -1), (15, len(dens) + 7)):
        bad = rows.clone()
        bad[777, col] = value
        with pytest.raises(hopgpu.HopError) as e:
            h.hop_link(dens, bad, 16)
        assert e.value.code == hopgpu.HOP_EINVAL
