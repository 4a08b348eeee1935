"""Curl and Phi of the FP64 passes at the edges of their range: fields whose values come near the smallest
doubles, and components of very different size, on grids of the fixed-point passes (an axis above 32)
and of the native ones.

Tolerances: those of the passes' own tests, 4e-15 (fixed point) and 1.6e-14 (native) of the largest value; the
spacing of subnormal results, 2^-1074, is at most 2^-60 of the largest value here."""

import numpy as np
import pytest

import oracle as O
import scfft_inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1803_01346_gb300 as S  # noqa: E402
from paper_1803_01346_gb300 import build as B  # noqa: E402

L = (1.6, 1.3, 1.5)
GRIDS = [((48, 16, 64), 4e-15), ((16, 96, 32), 4e-15), ((32, 16, 32), 1.6e-14)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.build()


def context(n):
    ctx = S.Context(n, L)
    ctx.precompute_kernel()
    return ctx


def run(ctx, op, f):
    out = torch.empty(f.size, dtype=torch.float64, device="cuda")
    getattr(ctx, op)(torch.from_numpy(np.ascontiguousarray(f).ravel()).cuda(), out)
    torch.cuda.synchronize()
    return out.cpu().numpy().reshape(f.shape)


@pytest.mark.parametrize("n,tol", GRIDS)
def test_fields_near_the_smallest_doubles(n, tol):
    f = I.random_field((3,) + O.Grid(n, L).shape, 31)
    ctx = context(n)
    for op in ("curl", "phi"):
        a = run(ctx, op, f)
        for e in (-960, -980, -1000, -1010):
            b = np.ldexp(run(ctx, op, np.ldexp(f, e)), -e)
            assert np.abs(a - b).max() < tol * np.abs(a).max(), (op, e, np.abs(a - b).max() / np.abs(a).max())


@pytest.mark.parametrize("n,tol", GRIDS)
@pytest.mark.parametrize("large", [0, 1, 2])
def test_each_output_keeps_its_own_precision(n, tol, large):
    """One component a million times the others: the output that reads only the small ones is small."""
    g = O.Grid(n, L)
    f = I.random_field((3,) + g.shape, 32)
    f[[q for q in range(3) if q != large]] *= 1e-6
    ctx = context(n)
    for op, ref in (("curl", O.curl_s(f, g)), ("phi", O.phi_hockney(f, g))):
        got = run(ctx, op, f)
        for q in range(3):
            assert np.abs(got[q] - ref[q]).max() < tol * np.abs(ref[q]).max(), (op, q)


@pytest.mark.parametrize("n,tol", GRIDS)
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_a_large_gradient_leaves_the_rest_of_the_curl_alone(n, tol, axis):
    """Component a, 30 to a million times the others, varies along axis a only, or not at all: its curl is zero
    on every mode, so the curl is that of the others."""
    g = O.Grid(n, L)
    f = I.random_field((3,) + g.shape, 33)
    f[axis] = 0.0
    ctx = context(n)
    ref = run(ctx, "curl", f)
    line = I.random_field((n[axis],), 34).reshape([-1 if 2 - axis == d else 1 for d in range(3)])
    for big in (line, 1.0):
        for size in (30.0, 1e3, 1e6):
            h = f.copy()
            h[axis] = size * big
            got = run(ctx, "curl", h)
            assert np.abs(got - ref).max() < tol * np.abs(ref).max(), (size, np.abs(got - ref).max() / np.abs(ref).max())
