"""The native FP64 passes of small grids (every axis 16 or 32), whose transforms of 16, 32 and 64 points
lie across the lanes of a warp: curl and Phi on all eight grids against the oracle, components of very
different size, and an infinity.

Tolerance: a transform of up to 64 points adds at most 6 roundings of 2^-53 a value; twelve passes of
them (six here, six in the oracle), the curl's wavenumbers at most 8 times their mean, and a largest
value some 4 times the mean: 6 * 12 * 1.1e-16 * 8 / 4 = 1.6e-14 of the largest value."""

import itertools

import numpy as np
import pytest

import oracle as O
import scfft_inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1803_01346_gb300 as S  # noqa: E402
from paper_1803_01346_gb300 import build as B  # noqa: E402

TOL = 1.6e-14
L = (1.6, 1.3, 1.5)


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.build()


def run(ctx, op, f, shape):
    out = torch.empty(f.size, dtype=torch.float64, device="cuda")
    getattr(ctx, op)(torch.from_numpy(np.ascontiguousarray(f).ravel()).cuda(), out)
    torch.cuda.synchronize()
    return out.cpu().numpy().reshape((3,) + shape)


@pytest.mark.parametrize("n", list(itertools.product((16, 32), repeat=3)))
@pytest.mark.parametrize("op", ["curl", "phi"])
def test_operators_match_the_oracle(n, op):
    g = O.Grid(n, L)
    f = I.random_field((3,) + g.shape, 21)
    ctx = S.Context(n, L)
    ctx.precompute_kernel()
    got = run(ctx, op, f, g.shape)
    ref = O.curl_s(f, g) if op == "curl" else O.phi_hockney(f, g)
    assert np.abs(got - ref).max() < TOL * np.abs(ref).max()
    # each component alone: the other two of its result come from it, its own is zero
    for q in range(3):
        e = np.zeros_like(f)
        e[q] = f[q]
        one = run(ctx, op, e, g.shape)
        assert not one[q].any()
        f2 = f.copy()
        f2[q] = 0.0
        rest = run(ctx, op, f2, g.shape)
        assert np.abs(one + rest - got).max() < TOL * np.abs(got).max()


@pytest.mark.parametrize("n", [(16, 16, 16), (32, 16, 32)])
def test_an_infinity_reaches_what_reads_it(n):
    g = O.Grid(n, L)
    f = I.random_field((3,) + g.shape, 22)
    f[1, 5, 7, 9] = np.inf
    ctx = S.Context(n, L)
    ctx.precompute_kernel()
    for op in ("curl", "phi"):
        got = run(ctx, op, f, g.shape)
        assert not np.isfinite(got[0]).any() and not np.isfinite(got[2]).any() and np.isfinite(got[1]).all(), op
