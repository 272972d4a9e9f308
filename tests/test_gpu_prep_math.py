"""The preparation's FP64 functions against quad precision (numpy long double)
and CUDA's own results, and the records they give over the raw parameters'
range.

Bounds, in units in the last place of the result (u = 2^-53 relative):
  exp        half an ulp for the last addition, at most 0.05 for the
             polynomial's and the reduction's roundings and its remainder
  sigmoid    1 / (1 + e): 0.5 for the quotient, 1 for the rounding of 1 + e
             and 2 * 0.52 for e's own error, each relative to a result just
             below a power of two
  2 s - 1    absolute: for a sigmoid near 1, (0.5 + 0.52 + 0.5) 2^-53 from
             1 + e and the quotient, doubled and with the quotient's half ulp
             on the other side of 1: 2 * 2.04 * 2^-53
  a / b      equal to the division
"""
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


def both(ndg, which, a, b=None):
    import torch
    put = lambda v: None if v is None else torch.as_tensor(v, dtype=torch.float64).cuda()  # noqa: E731
    own, cuda = ndg.selftest_math(which, put(a), put(b))
    return own.cpu().numpy(), cuda.cpu().numpy()


def ulps(got, ref):
    _, e = np.frexp(ref.astype(np.float64))
    return float((np.abs(got.astype(np.longdouble) - ref) / np.ldexp(1.0, e - 53)).max())


def arguments(seed):
    """FP32 values: the whole normal range, the 64 table entries of several
    binades, values about one and tiny ones, both sides of the range's end."""
    r = synth.rng(seed)
    k = np.arange(-64 * 12, 64 * 12) * np.log(2) / 64
    v = np.concatenate([r.uniform(-689, 689, 300_000), r.uniform(-20, 20, 300_000), r.uniform(-1, 1, 300_000),
                        np.exp(r.uniform(np.log(1e-12), np.log(90), 300_000)) * r.choice([-1, 1], 300_000),
                        k, k + 0.00541, k - 0.00541, [0.0, -0.0, 1e-45, -1e-45, 1e-38, 689.99, 690.0, -690.0]])
    return v.astype(np.float32).astype(np.float64)


def test_exp_is_within_its_bound_and_cudas_error(ndg):
    v = arguments(1)
    own, cuda = both(ndg, 0, v)
    ref = np.exp(v.astype(np.longdouble))
    e, c = ulps(own, ref), ulps(cuda, ref)
    print(f"exp: {e:.4f} ulp, CUDA's {c:.4f}")
    assert e <= 0.55 and e <= c


def test_sigmoid_and_off_diagonal_are_within_their_bounds(ndg):
    v = arguments(2)
    x = v.astype(np.longdouble)
    own, cuda = both(ndg, 1, v)
    ref = 1 / (1 + np.exp(-x))
    e = ulps(own, ref)
    own2, cuda2 = both(ndg, 2, v)
    d = float(np.abs(own2.astype(np.longdouble) - np.tanh(x / 2)).max())
    print(f"sigmoid: {e:.4f} ulp, CUDA's {ulps(cuda, ref):.4f}; 2 s - 1: {d:.3e}")
    assert e <= 2.54
    assert d <= 2 * 2.04 * 2.0 ** -53
    # where a coefficient is not tiny, the FP32 value is the one CUDA's functions give
    big = np.abs(v) >= 1e-7
    assert np.array_equal(own2[big].astype(np.float32), cuda2[big].astype(np.float32))


def test_functions_outside_the_normal_range_are_cudas(ndg):
    v = np.array([690.0, 700.0, 709.5, 709.9, 1e4, 3e38, np.inf, -690.0, -700.0, -745.0, -746.0, -1e4, -np.inf, np.nan])
    for which in (0, 1, 2):
        own, cuda = both(ndg, which, v)
        assert np.array_equal(own, cuda, equal_nan=True), which


def test_quotients_equal_the_division(ndg):
    r = synth.rng(4)
    n = 500_000
    sign = r.choice([-1.0, 1.0], n)
    a = np.ldexp(r.uniform(1, 2, n), r.integers(-400, 400, n)) * sign
    b = np.ldexp(r.uniform(1, 2, n), r.integers(-400, 400, n))
    # quotients next to the midpoint of two FP64 numbers
    a = np.concatenate([a, 1 + r.integers(0, 50, n) * 2.0 ** -52])
    b = np.concatenate([b, 2 - r.integers(1, 50, n) * 2.0 ** -52])
    own, cuda = both(ndg, 3, a, b)
    assert np.array_equal(own, cuda)


def test_records_over_the_range_of_all_raw_parameters(ndg, oracle):
    """Brightness, colours and children far out on both sides: the lists and
    the FP32 form's outputs are the oracle's."""
    import torch
    N, G, Q, tile, k = 4, 1500, 2048, 64, 8
    r = synth.rng(70)
    mix, ch = synth.mixture(N, G, 71), synth.children(N, G, 72)
    far = lambda s, *sh: (r.choice([1e-4, 0.3, 3.0, 30.0, 750.0], sh) * r.choice([-1.0, 1.0], sh) * s).astype(np.float32)  # noqa: E731
    mix["alpha_raw"] = r.uniform(-60, 3, G).astype(np.float32)
    mix["color_raw"], ch["c_color_raw"] = far(1, G, 3), far(1, G, 3)
    ch["c_alpha_raw"] = r.uniform(-60, 1, G).astype(np.float32)
    i, j = np.tril_indices(N)
    ch["u_theta"] = np.where(i == j, r.uniform(-3, 1, (G, len(i))), far(1, G, len(i))).astype(np.float32)
    ch["m_u"] = r.uniform(-4, 4, (G, N)).astype(np.float32)
    x = synth.queries_box(N, Q, 73)
    gm = ndg.Mixture.from_arrays(N, mix, ch)
    proj = synth.projections(N, k, 74)
    cp = ndg.CullParams(k, torch.as_tensor(proj).cuda(), 1 / 255, 3.0, 64)
    ev = ndg.Evaluator(gm, torch.as_tensor(x).cuda(), tile, cp, backward=False)
    E = ev.build(gm)
    L, m, w = oracle.activate(oracle_raw(oracle, mix, ch))
    offs, ids = oracle.cull_contract(L, m, w, x.astype(np.float64), tile, proj, 1 / 255, 3.0, 64)
    assert E == offs[-1] > 0
    got = csr_sets(ev.cull.offsets.cpu().numpy(), ev.cull.ids[:E].cpu().numpy())
    for t, (a, b) in enumerate(zip(got, csr_sets(offs, ids))):
        assert np.array_equal(a, b), f"tile {t}"
    yo = oracle.eval(L, m, w, x.astype(np.float64), tile, offs, ids)
    assert_outputs_close(ev.forward(gm).cpu().numpy(), yo)
    assert ndg.read_status(ev.ws) == 0


@pytest.mark.parametrize("theta", [-80.0, 85.0])
def test_records_at_the_ends_of_the_fp32_range(ndg, oracle, theta):
    """One diagonal at e^-80 (such Gaussians contribute nothing) or e^85 (a
    flat direction)."""
    import torch
    N, G, Q, tile = 3, 64, 512, 64
    mix = synth.mixture(N, G, 80)
    mix["theta"][::2, 0] = theta
    x = synth.queries_box(N, Q, 81)
    gm = ndg.Mixture.from_arrays(N, mix)
    ev = ndg.Evaluator(gm, torch.as_tensor(x).cuda(), tile, ndg.CullParams(0, None, 0.0, 3.0, 1), backward=False)
    ev.build(gm)
    L, m, w = oracle.activate(oracle_raw(oracle, mix))
    assert_outputs_close(ev.forward(gm).cpu().numpy(), oracle.eval(L, m, w, x.astype(np.float64)))
