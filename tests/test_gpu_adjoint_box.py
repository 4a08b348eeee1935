"""The transposed iteration keeps Phi's result and the curl's input to the solid's bounding box: one
right-hand side's vector-Jacobian product for an off-centre solid whose box starts at an odd row and
plane, against the oracle, on a context whose buffers hold large values of earlier calls (so that a
row or plane that is read without having been written shows).

Tolerances: those of the reverse mode everywhere, 1e-10 in FP64 and 1e-4 in FP32."""

import numpy as np
import pytest

import oracle as O
import scfft_inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1803_01346_gb300 as S  # noqa: E402
from paper_1803_01346_gb300 import build as B  # noqa: E402

L = (1.0, 1.4, 0.8)


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.build()


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64).ravel()).cuda()


@pytest.mark.parametrize("prec,tol", [(S.PREC_F64, 1e-10), (S.PREC_DF64, 1e-10), (S.PREC_F32, 1e-4)])
@pytest.mark.parametrize("n", [(16, 32, 16), (32, 16, 32), (32, 48, 64), (64, 32, 16), (48, 96, 32), (16, 16, 128)])
def test_vjp_of_an_off_centre_solid_matches_the_oracle(n, prec, tol):
    K = 3
    g = O.Grid(n, L)
    mask = np.zeros(g.shape, dtype=bool)
    mask[3:9, 5:12, 2:n[0] - 6] = True
    mask[5, 7, 4] = False
    path = ([0.0, 1.0], [[0, 0, 0], [0.3, -0.2, 0.9]])
    jc = I.jc_noise(g.shape, 5)
    ctx = S.Context(n, L, n_power=7.0, rho_out=5.0, precision=prec, delta_it=0.0, max_iter=K)
    ctx.set_geometry(mask)
    ctx.set_field_path(*path)
    ctx.set_jc_map(dev(jc))
    ctx.precompute_kernel()
    prob = O.Problem(g, mask, O.Material(n=7.0, rho_out=5.0, jc=jc), O.FieldPath(*path))
    rng = np.random.default_rng(3)
    h = O.phi_hockney(O.curl_s(0.5 * rng.standard_normal((3,) + g.shape), g) * mask, g) + 0.05
    lam = rng.standard_normal(h.shape)
    big, out = dev(1e6 * rng.standard_normal(h.shape)), torch.empty(h.size, dtype=torch.float64, device="cuda")
    ctx.phi(big, out)
    ctx.curl(big, out)
    ref = O.rhs_vjp(prob, 0.4, h, lam, K)
    mu_h, mu_g = torch.empty_like(out), torch.empty_like(out)
    mu_jc = torch.empty(h.size // 3, dtype=torch.float64, device="cuda")
    mu_a = ctx.rhs_vjp(dev(h), dev(lam), mu_h, mu_g, mu_jc)
    torch.cuda.synchronize()
    for got, want in ((mu_h, ref.mu_h), (mu_g, ref.mu_g), (mu_jc, ref.mu_jc)):
        got = got.cpu().numpy().reshape(want.shape)
        assert np.abs(got - want).max() < tol * np.abs(want).max()
    assert np.abs(np.array(mu_a) - ref.mu_a).max() < tol * np.abs(ref.mu_a).max()
