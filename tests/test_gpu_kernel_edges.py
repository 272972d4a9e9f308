"""Edges of the kernels' own layouts: chunks of 96 candidates and 32-candidate
builder groups of the tensor-core forward, groups of tiles and the two byte
compares of the cull's count pass, and the preparation's exponentials over the
range of the raw parameters."""
import numpy as np
import pytest

from helpers import assert_outputs_close, csr_sets, oracle_raw
from paper_2405_20067_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ndg():
    import torch
    from paper_2405_20067_gb300 import build, ndg as _ndg
    build.build()
    assert torch.cuda.is_available(), "GPU tests need a GPU"
    return _ndg


def setup(ndg, N, mix, x, tile, k, cutoff, B, seed):
    import torch
    gm = ndg.Mixture.from_arrays(N, mix)
    proj = synth.projections(N, k, seed) if k else None
    cp = ndg.CullParams(k, torch.as_tensor(proj).cuda() if k else None, cutoff, 3.0, B)
    ev = ndg.Evaluator(gm, torch.as_tensor(x).cuda(), tile, cp, backward=False)
    return gm, proj, ev, ev.build(gm)


@pytest.mark.parametrize("N", [2, 6, 8, 9, 10, 12])
@pytest.mark.parametrize("G", [1, 32, 33, 95, 96, 97, 769])
def test_tc_forward_at_chunk_and_group_edges(ndg, oracle, N, G):
    """Every Gaussian a candidate of every tile (k = 0); tiles of one and of
    two row blocks, the last one ragged."""
    mix = synth.mixture(N, G, 40 + N)
    x = synth.queries_box(N, 600, 41)
    L, m, w = oracle.activate(oracle_raw(oracle, mix))
    yo = oracle.eval(L, m, w, x.astype(np.float64))
    for tile in (256, 128):
        gm, _, ev, E = setup(ndg, N, mix, x, tile, 0, 0.0, 1, 0)
        assert E == -(-600 // tile) * G
        y = ev.forward(gm, mode=ndg.NDG_MODE_TC).cpu().numpy()
        assert_outputs_close(y, yo, rtol=1e-3, floor=1e-3)
        assert ndg.read_status(ev.ws) == 0


# tiles: below and at the two switches of the tiles per CTA (1216 and 2432),
# and counts that are no multiple of them; buckets: both byte compares
@pytest.mark.parametrize("T,B", [(1215, 64), (1217, 64), (2432, 128), (2435, 64), (2435, 129), (2435, 255), (1217, 200)])
@pytest.mark.parametrize("k", [3, 16])
def test_cull_lists_by_tile_group_and_buckets(ndg, oracle, T, B, k):
    N, G, tile = 5, 400, 8
    mix = synth.mixture(N, G, 50)
    x = synth.queries_box(N, T * tile - 3, 51)
    _, proj, ev, E = setup(ndg, N, mix, x, tile, k, 1 / 255, B, 52)
    L, m, w = oracle.activate(oracle_raw(oracle, mix))
    offs, ids = oracle.cull_contract(L, m, w, x.astype(np.float64), tile, proj, 1 / 255, 3.0, B)
    assert E == offs[-1] and 0 < E < T * G
    assert np.array_equal(ev.cull.offsets.cpu().numpy(), offs)
    got = csr_sets(ev.cull.offsets.cpu().numpy(), ev.cull.ids[:E].cpu().numpy())
    for t, (a, b) in enumerate(zip(got, csr_sets(offs, ids))):
        assert np.array_equal(a, b), f"tile {t}"


def test_preparation_over_the_range_of_the_raw_parameters(ndg, oracle):
    """Off-diagonals from far inside both saturated ends, widths over e^+-9:
    the lists (FP32-rounded activations) are the oracle's."""
    N, G, Q, tile, k = 4, 2000, 4096, 64, 8
    r = synth.rng(60)
    mix = synth.mixture(N, G, 61)
    i, j = np.tril_indices(N)
    th = np.where(i == j, r.uniform(-9, 2, (G, len(i))), r.choice([1e-3, 0.5, 5.0, 40.0, 800.0], (G, len(i)))
                  * r.choice([-1.0, 1.0], (G, len(i))))
    mix["theta"] = th.astype(np.float32)
    x = synth.queries_box(N, Q, 62)
    _, proj, ev, E = setup(ndg, N, mix, x, tile, k, 1 / 255, 64, 63)
    L, m, w = oracle.activate(oracle_raw(oracle, mix))
    offs, ids = oracle.cull_contract(L, m, w, x.astype(np.float64), tile, proj, 1 / 255, 3.0, 64)
    assert E == offs[-1]
    got = csr_sets(ev.cull.offsets.cpu().numpy(), ev.cull.ids[:E].cpu().numpy())
    for t, (a, b) in enumerate(zip(got, csr_sets(offs, ids))):
        assert np.array_equal(a, b), f"tile {t}"
