"""Counts around the limits of the one-block sort (2,048 and 8,192 pairs): the
particle sort, the boundary list and the group ranking go through it.  Lists,
boundaries, chains and groups against the oracle fed the GPU's densities;
equal boundary sums, so that the merge's tie order decides."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle
import paper_1001_3411_gb300 as hopgpu
import synth
from hop_parity import check_knn_rows, oracle_downstream

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hop():
    hopgpu.build_library()
    h = hopgpu.Hop(0)
    yield h
    h.close()


@pytest.mark.parametrize("n", [65, 511, 2047, 2048, 2049, 8191, 8192, 8193])
def test_particle_sort_and_groups(hop, n):
    pos = synth.nfw_box(n, 400 + n)[0] if n > 600 else synth.uniform_box(n, n)
    d = torch.from_numpy(pos).cuda()
    p = hopgpu.default_params()
    r = hop.hop_run(d, p, ld_nbr=16, want_chain=True)
    b = hop.hop_run_batch(d, [0, n], [1.0], p, ld_nbr=16)
    for key in ("dens", "nbr", "group"):
        assert torch.equal(r[key], b[key]), key
    nbr, dens = r["nbr"].cpu().numpy(), r["dens"].cpu().numpy()
    q = np.arange(0, n, 3)
    check_knn_rows(pos, nbr[q], q, 64, name=str(n))
    o = oracle_downstream(dens, nbr, 16, 4, 80.0, 200.0, 240.0)
    assert np.array_equal(r["chain"].cpu().numpy(), o["chain"])
    assert np.array_equal(r["group"].cpu().numpy(), o["group"]) and r["n_groups"] == o["n_groups"]


@pytest.mark.parametrize("chains", [60, 1500, 6000])
@pytest.mark.parametrize("mutual", [False, True])
def test_boundaries_and_merge_of_many_chains(hop, chains, mutual):
    """Random chain graphs with densities on a 0.1 grid: many equal sums."""
    n, n_merge = 40000, 4
    chain, dens, rows = synth.chain_graph_case(n, n_merge, chains, 5 + chains, mutual)
    dens = dens.astype(np.float32).astype(np.float64)     # the densities the GPU holds
    d_o, d_s, d_p = 60.0, 200.0, 420.0
    ct, dt = torch.from_numpy(chain).cuda(), torch.from_numpy(dens.astype(np.float32)).cuda()
    pair, s = hop.hop_boundaries(ct, dt, torch.from_numpy(rows).cuda(), n_merge, d_o)
    lo, hi, s_o = oracle.boundaries(chain, dens, rows, n_merge, d_o)
    pr = pair.cpu().numpy()
    assert np.array_equal(pr >> 32, lo) and np.array_equal(pr & 0xFFFFFFFF, hi) and np.array_equal(s.cpu().numpy(), s_o)
    group, ng = hop.hop_merge(ct, dt, pair, s, d_o, d_s, d_p)
    g_o, ng_o = oracle.merge(chain, dens, lo, hi, s_o, d_o, d_s, d_p)
    assert ng == ng_o and np.array_equal(group.cpu().numpy(), g_o)
