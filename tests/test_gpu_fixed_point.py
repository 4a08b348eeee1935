"""The 64-bit fixed-point passes of the FP64 path (grids with an axis above 32) at their edges: every
transform length (16 to 128 unpadded, 32 to 256 padded) on grids whose axes differ, ragged column
tiles, exact invariance under a power-of-two scale over FP64's range, components of very different
size, and a NaN.

Tolerance: a pass rounds its results to doubles (relative error 2^-53 of each) and its transform
adds less; six passes, with the curl's wavenumbers at most 8 times their mean, and the oracle's own
FP64 transforms of the same size stay below 4e-15 of the largest value."""

import numpy as np
import pytest

import oracle as O
import scfft_inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1803_01346_gb300 as S  # noqa: E402
from paper_1803_01346_gb300 import build as B  # noqa: E402

TOL = 4e-15
L = (1.6, 1.3, 1.5)


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.build()


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64).ravel()).cuda()


def run(ctx, op, f, shape):
    out = torch.empty(f.size, dtype=torch.float64, device="cuda")
    getattr(ctx, op)(dev(f), out)
    torch.cuda.synchronize()
    return out.cpu().numpy().reshape((3,) + shape)


@pytest.mark.parametrize("n", [(16, 32, 48), (64, 96, 16), (128, 16, 32), (48, 128, 64), (96, 48, 128), (32, 64, 96)])
@pytest.mark.parametrize("op", ["curl", "phi"])
def test_operators_match_the_oracle(n, op):
    g = O.Grid(n, L)
    f = I.random_field((3,) + g.shape, 11)
    f[2] *= 1e-6  # one component far below the others: each output keeps its own precision
    ctx = S.Context(n, L)
    ctx.precompute_kernel()
    got = run(ctx, op, f, g.shape)
    ref = O.curl_s(f, g) if op == "curl" else O.phi_hockney(f, g)
    for q in range(3):
        assert np.abs(got[q] - ref[q]).max() < TOL * np.abs(ref[q]).max(), (q, np.abs(got[q] - ref[q]).max())


@pytest.mark.parametrize("e", [-900, -200, 300, 900])
def test_a_power_of_two_scale_is_exact(e):
    n = (48, 16, 64)
    g = O.Grid(n, L)
    f = I.random_field((3,) + g.shape, 12)
    ctx = S.Context(n, L)
    ctx.precompute_kernel()
    for op in ("curl", "phi"):
        a, b = run(ctx, op, f, g.shape), run(ctx, op, np.ldexp(f, e), g.shape)
        assert np.array_equal(np.ldexp(a, e), b), op


def test_a_zero_field_and_a_lone_component():
    n = (32, 48, 16)
    g = O.Grid(n, L)
    ctx = S.Context(n, L)
    ctx.precompute_kernel()
    z = np.zeros((3,) + g.shape)
    assert not run(ctx, "curl", z, g.shape).any() and not run(ctx, "phi", z, g.shape).any()
    z[1] = I.random_field(g.shape, 13)
    for op, ref in (("curl", O.curl_s(z, g)), ("phi", O.phi_hockney(z, g))):
        got = run(ctx, op, z, g.shape)
        assert np.abs(got - ref).max() < TOL * np.abs(ref).max()


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_a_value_that_is_no_number_makes_its_outputs_nan(bad):
    n = (48, 32, 64)
    g = O.Grid(n, L)
    f = I.random_field((3,) + g.shape, 14)
    f[1, 5, 7, 9] = bad
    ctx = S.Context(n, L)
    ctx.precompute_kernel()
    for op in ("curl", "phi"):
        got = run(ctx, op, f, g.shape)
        # components x and z read the y component; y does not
        assert np.isnan(got[0]).all() and np.isnan(got[2]).all() and np.isfinite(got[1]).all(), op
