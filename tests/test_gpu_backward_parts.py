"""The backward with a tile's candidates in several parts and in one: the same
bits, at list lengths on both sides of the chunks' and the parts' edges; and
lists of many chunks in one CTA against the oracle (the reuse of every stage,
stash slot and accumulator).  A launch of a few tiles is split; the same tiles
followed by empty ones are not (the rule goes by the average list)."""
import numpy as np
import pytest

from helpers import NAMES, assert_grads_close, oracle_raw
from paper_2405_20067_gb300 import synth

pytestmark = pytest.mark.gpu
TILE = 256
EMPTY = 600  # empty tiles behind the others: less than a chunk per tile on average


@pytest.fixture(scope="module")
def ndg():
    import torch
    from paper_2405_20067_gb300 import build, ndg as _ndg
    build.build()
    assert torch.cuda.is_available(), "GPU tests need a GPU"
    return _ndg


def lists(G, lengths, extra, seed):
    """Ascending ids, `lengths[t]` of G in tile t, and `extra` empty tiles."""
    r = synth.rng(seed)
    ids = [np.sort(r.choice(G, n, replace=False)) for n in lengths]
    offs = np.concatenate([[0], np.cumsum([len(i) for i in ids]), np.full(extra, sum(lengths))]).astype(np.int64)
    return offs, np.concatenate(ids).astype(np.int32)


def backward(ndg, N, mix, x, dy, offs, ids, mode, cap=None):
    """Gradients for the first rows of x and dy (ragged last tile), on given lists."""
    import torch
    T = len(offs) - 1
    gm = ndg.Mixture.from_arrays(N, mix)
    xt, dt = torch.as_tensor(x).cuda(), torch.as_tensor(dy).cuda()
    c = ndg.Cull(T, cap or max(len(ids), 1))
    c.offsets.copy_(torch.as_tensor(offs))
    c.ids[:len(ids)] = torch.as_tensor(ids).cuda()
    c.E_dev.fill_(len(ids))
    ws = ndg.workspace(ndg.workspace_size(gm, xt, TILE, None, c.E_cap))
    g = gm.zeros_like()
    ndg.backward(gm, xt, TILE, c, dt, g, ws, mode=mode)
    assert ndg.read_status(ws) == 0
    return [getattr(g, n).cpu().numpy() for n in NAMES[:4]]


def inputs(N, G, T, extra, seed):
    """T tiles of queries, then `extra` more."""
    mix = synth.mixture(N, G, seed)
    x = np.concatenate([synth.queries_box(N, T * TILE, seed + 1), synth.queries_box(N, extra * TILE, seed + 2)])
    dy = (synth.rng(seed + 3).standard_normal((len(x), 3)) / (3 * len(x))).astype(np.float32)
    return mix, x, dy


@pytest.mark.parametrize("mode", ["tc", "fp32"])
@pytest.mark.parametrize("N", [1, 3, 6, 7, 8, 9, 10, 11, 12])
def test_parts_give_the_bits_of_one(ndg, N, mode):
    md, step = (ndg.NDG_MODE_TC, 128) if mode == "tc" else (ndg.NDG_MODE_FP32, 256)
    lengths = [1, step - 1, step, step + 1, 2 * step - 1, 2 * step, 2 * step + 1, 0, 3 * step, 5 * step + 7,
               8 * step - 1, 8 * step, 8 * step + 1, 11 * step]
    G, T = 11 * step, len(lengths)
    mix, x, dy = inputs(N, G, T, EMPTY, 500 + N)
    offs, ids = lists(G, lengths, EMPTY, 510 + N)
    whole = backward(ndg, N, mix, x, dy, offs, ids, md)
    split = backward(ndg, N, mix, x[:T * TILE], dy[:T * TILE], offs[:T + 1], ids, md)
    for n, a, b in zip(NAMES, split, whole):
        assert np.abs(b).max() > 0 and np.array_equal(a, b), n
    # a capacity far above the lists asks for more parts than a tile has steps
    roomy = backward(ndg, N, mix, x[:T * TILE], dy[:T * TILE], offs[:T + 1], ids, md, cap=40 * len(ids))
    for n, a, b in zip(NAMES, roomy, whole):
        assert np.array_equal(a, b), n


@pytest.mark.parametrize("N", [3, 6, 7, 8, 9, 10, 11, 12])
def test_many_chunks_in_one_cta_match_the_oracle(ndg, oracle, N):
    """10 chunks of two query units and 7 of one (a tile of 100 queries last)."""
    lengths, G = [9 * 128 + 5, 7 * 128 - 3], 1300
    mix, x, dy = inputs(N, G, 2, EMPTY, 600 + N)
    # the short tile last: the empty tiles come first
    x, dy = np.roll(x, EMPTY * TILE, axis=0)[:-156], np.roll(dy, EMPTY * TILE, axis=0)[:-156]
    offs, ids = lists(G, lengths, 0, 610 + N)
    offs = np.concatenate([np.zeros(EMPTY, np.int64), offs])
    got = dict(zip(NAMES, backward(ndg, N, mix, x, dy, offs, ids, ndg.NDG_MODE_TC)))
    want = oracle.grad(oracle_raw(oracle, mix), x.astype(np.float64), TILE, offs, ids, dy.astype(np.float64))
    assert_grads_close(got, want, NAMES[:4], rtol=1e-3)
