"""Subhalos at several thresholds at once: numbers of thresholds around the
eight handled together, in any order and repeated, chains in runs of every
length along the particle order, and rows that do not start on 16 bytes,
against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle
import paper_1001_3411_gb300 as hopgpu
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hop():
    hopgpu.build_library()
    h = hopgpu.Hop(0)
    yield h
    h.close()


def _check(hop, chain, dens, rows, n_merge, d_o, levels, n_min=1):
    dens = dens.astype(np.float32).astype(np.float64)
    sub, n_sub = hop.hop_subhalos(torch.from_numpy(chain).cuda(), torch.from_numpy(dens.astype(np.float32)).cuda(),
                                  torch.from_numpy(np.ascontiguousarray(rows)).cuda(), n_merge, d_o, levels, n_min)
    sub_o, n_o = oracle.adaptahop(chain, dens, rows, n_merge, d_o, [float(np.float32(x)) for x in levels], n_min, 0.0)
    assert n_sub.tolist() == n_o.tolist()
    assert np.array_equal(sub.cpu().numpy(), sub_o)


@pytest.mark.parametrize("count", [1, 7, 8, 9, 17])
def test_numbers_of_thresholds(hop, count):
    chain, dens, rows = synth.chain_graph_case(20012, 4, 1500, 40 + count, True)
    levels = np.random.default_rng(count).choice([80.0, 95.5, 120.0, 180.0, 260.0, 500.0], count).tolist()
    _check(hop, chain, dens, rows, 4, 80.0, levels, n_min=2)


@pytest.mark.parametrize("run", [1, 3, 31, 32, 33, 64, 1024, 5000])
@pytest.mark.parametrize("n_merge", [3, 5])
def test_runs_of_members(hop, run, n_merge):
    """Particle order sorted so that each chain's members come in runs of
    `run` consecutive particles."""
    chain, dens, rows = synth.chain_graph_case(20000, n_merge, 40, run, True)
    by_chain = np.argsort(chain, kind="stable")
    within = np.empty(len(chain), dtype=np.int64)
    _, start, size = np.unique(chain[by_chain], return_index=True, return_counts=True)
    within[by_chain] = np.arange(len(chain)) - np.repeat(start, size)
    new = np.lexsort((within, chain, within // run))      # old index of the particle at each place
    place = np.empty(len(chain), dtype=np.int64)
    place[new] = np.arange(len(chain))
    _check(hop, place[chain[new]].astype(np.int32), dens[new], place[rows[new]].astype(np.int32), n_merge, 70.0,
           [70.0, 150.0, 300.0])
