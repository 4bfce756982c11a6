"""Calls in a GPU memory that is almost full: scratch that only speeds a call
up must not make it fail.  Each call runs once with room, then again on a new
context with the room taken away, and must give the same result."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1001_3411_gb300 as hopgpu

pytestmark = pytest.mark.gpu
MB = 1 << 20


def _fill(leave):
    """All but `leave` bytes of the free device memory."""
    torch.cuda.synchronize()
    return torch.empty(torch.cuda.mem_get_info()[0] - leave, dtype=torch.uint8, device="cuda")


@pytest.mark.parametrize("f64,n,leave", [(True, 4000037, 48 * MB), (False, 8000009, 24 * MB)])
def test_density_without_room_for_the_boxes(f64, n, leave):
    """The grouped kNN's float copies (64 MB here), boxes (18 or 37 MB) and
    lists (20 or 32 MB) do not fit: the single-scan kernel serves the call."""
    hopgpu.build_library()
    g = torch.Generator(device="cuda").manual_seed(3)
    pos = torch.rand(n, 3, generator=g, device="cuda", dtype=torch.float64 if f64 else torch.float32)
    p = hopgpu.default_params(pos_is_f64=int(f64), radius_mode=hopgpu.HOP_RADIUS_COUNT)
    hop = hopgpu.Hop(0)
    try:
        ref = hop.hop_density(pos, p, ld_nbr=16, want_rk=True)
    finally:
        hop.close()
    hop = hopgpu.Hop(0)
    hop.apply_tuning(8, 1, 4)      # the single-scan kernel: every other buffer of the call
    hop.hop_density(pos, p, ld_nbr=16, want_rk=True)   # (its results' memory is kept by torch)
    hop.apply_tuning(8, 1, 0)
    rest = _fill(leave)
    try:
        out = hop.hop_density(pos, p, ld_nbr=16, want_rk=True)
    finally:
        del rest
        hop.close()
        torch.cuda.empty_cache()
    for x, y, name in zip(out, ref, ("nbr", "dens", "rk")):
        assert torch.equal(x, y), name


@pytest.mark.parametrize("eager", [False, True])
def test_batched_pass_without_room_for_the_boxes(eager):
    """The same for two subvolumes in one pass, captured or enqueued."""
    hopgpu.build_library()
    n = 8000009
    g = torch.Generator(device="cuda").manual_seed(5)
    pos = torch.rand(n, 3, generator=g, device="cuda")
    off, boxes = [0, 3000001, n], [1.0, 1.0]
    p = hopgpu.default_params(radius_mode=hopgpu.HOP_RADIUS_COUNT)
    hop = hopgpu.Hop(0)
    try:
        ref = hop.hop_run_batch(pos, off, boxes, p, ld_nbr=16, eager=eager)
    finally:
        hop.close()
    hop = hopgpu.Hop(0)
    hop.apply_tuning(8, 1, 4)
    hop.hop_run_batch(pos, off, boxes, p, ld_nbr=16, eager=eager)
    hop.apply_tuning(8, 1, 0)
    rest = _fill(24 * MB)
    try:
        out = hop.hop_run_batch(pos, off, boxes, p, ld_nbr=16, eager=eager)
    finally:
        del rest
        hop.close()
        torch.cuda.empty_cache()
    for key in ("dens", "group", "nbr"):
        assert torch.equal(out[key], ref[key]), key


def test_subhalos_without_room_for_eight_thresholds():
    """Arrays for eight thresholds at once (about 0.35 kB per chain) do not
    fit, those for fewer do."""
    hopgpu.build_library()
    rng = np.random.default_rng(4)
    n, n_chains = 2000000, 400000
    chain = rng.integers(0, n_chains, n).astype(np.int32)
    chain[:n_chains] = np.arange(n_chains)
    dens = (100.0 + rng.random(n) * 1000.0).astype(np.float32)
    dens[:n_chains] = (1200.0 + rng.permutation(n_chains) * 1e-3).astype(np.float32)
    nbr = rng.integers(0, n, (n, 4)).astype(np.int32)
    levels = [100.0 + 100.0 * i for i in range(8)]
    dev = [torch.from_numpy(x).cuda() for x in (chain, dens, nbr)]
    hop = hopgpu.Hop(0)
    try:
        sub, n_sub = hop.hop_subhalos(*dev, 4, 100.0, levels)
    finally:
        hop.close()
    hop = hopgpu.Hop(0)
    hop.hop_subhalos(*dev, 4, 100.0, levels[:1])   # every other buffer of the call
    again = torch.empty_like(sub)
    del again                                      # kept by torch for the labels below
    rest = _fill(48 * MB)
    try:
        out, n_out = hop.hop_subhalos(*dev, 4, 100.0, levels)
    finally:
        del rest
        hop.close()
        torch.cuda.empty_cache()
    assert torch.equal(out, sub) and np.array_equal(n_out, n_sub)
