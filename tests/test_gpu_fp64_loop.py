"""The FP64 Eq. 5 loop with an early stop runs as a captured graph; while profiling the host drives the same
passes.  Both give the same dh/dt bit for bit and the same iteration count, with either curl, again
after a change of geometry, and within one iteration of the oracle; and a step taken with each is the same."""

import numpy as np
import pytest

import oracle as O
import scfft_inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1803_01346_gb300 as S  # noqa: E402
from paper_1803_01346_gb300 import build as B  # noqa: E402

L = (1.0, 1.0, 1.0)


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.build()


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64).ravel()).cuda()


@pytest.mark.parametrize("n", [(16, 16, 32), (48, 32, 16)])
@pytest.mark.parametrize("curl", [S.CURL_SPECTRAL, S.CURL_FD])
def test_graph_loop_equals_host_loop(n, curl):
    g = O.Grid(n, L)
    path = ([0.0, 1.0], [[0, 0, 0], [0.3, -0.2, 0.9]])
    ctx = S.Context(n, L, n_power=20.0, rho_out=20.0, delta_it=2e-5, max_iter=50)
    ctx.set_field_path(*path)
    for mask in (I.cube(n, L, 1.0), I.sphere(n, L, 0.6)):
        ctx.set_geometry(mask)
        ctx.precompute_kernel()
        if curl != S.CURL_SPECTRAL:
            ctx.set_curl(curl)
        prob = O.Problem(g, mask, O.Material(n=20.0, rho_out=20.0), O.FieldPath(*path))
        jr = O.curl_s(I.random_field((3,) + g.shape, 4, 0.3), g) * mask[None]
        h = O.phi_hockney(jr, g)
        g0 = np.broadcast_to(prob.path.hedot(0.5)[:, None, None, None], h.shape).copy()
        out, steps = [], []
        for host in (True, False, False):
            ctx.profile(host)
            hd = torch.empty(h.size, dtype=torch.float64, device="cuda")
            i0 = ctx.stats()["iterations"]
            it = ctx.rhs(0.5, dev(h), dev(g0), hd)
            assert ctx.stats()["iterations"] - i0 == it
            out.append((it, hd.cpu().numpy()))
            hs, ws = dev(h), dev(g0)
            steps.append((ctx.step(0.5, 1e-4, 1.0, hs, ws)[:2], hs.cpu().numpy(), ws.cpu().numpy()))
            ctx.profile(False)
        for (it, v), (td, hs, ws) in zip(out[1:], steps[1:]):
            assert it == out[0][0] and np.array_equal(v, out[0][1])
            assert td == steps[0][0] and np.array_equal(hs, steps[0][1]) and np.array_equal(ws, steps[0][2])
        if curl == S.CURL_SPECTRAL:
            assert abs(out[0][0] - O.rhs(prob, 0.5, h, g0, delta_it=2e-5, max_iter=50).iters) <= 1
