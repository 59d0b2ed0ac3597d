"""Controls and terminal fields in the subnormal range of doubles are carried
with the bits that they hold."""
import numpy as np
import pytest

from paper_2602_14016_gb300 import synthetic

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

TINY = 2.0**-1035  # of unit fields: below the smallest normal double, 2^-1022
# What is held between passes has at least 20 bits there: the state rounds at
# 2^-1075, and its products with dt/6 (2^-13) and 1/n^2 (2^-16 at 256^2, then
# summed over n^2 modes of random sign) are 2^-1050 or more.
TOL = 2.0**-18


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.fail("a GPU test ran without a GPU")
    from paper_2602_14016_gb300 import api as A, build

    build.build()
    return A


def cu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def rel(a, b):
    """Relative difference of a = TINY b, taken at b's magnitude."""
    a = (torch.view_as_real(a) if a.is_complex() else a) * 2.0**600 * 2.0**435
    b = torch.view_as_real(b) if b.is_complex() else b
    return float(torch.linalg.norm(a - b) / torch.linalg.norm(b))


@pytest.mark.parametrize("n", [16, 64, 256])
@pytest.mark.parametrize("plain", [False, True])
def test_subnormal_fields_keep_their_bits(api, n, plain):
    ctx = api.Context(api.Config(n=n, nsteps=2, dt=1e-3, nu=1e-3, px=4, every=1))
    if plain:
        ctx.time_kernels("adj_cols")  # the plain sequence of pass kernels
    s = ctx.control_from_omega(cu(synthetic.random_vorticity_hat(n, 3)[None]))
    lam = cu(synthetic.unit_norm_terminal_hat(n, 4)[None])
    # the adjoint is linear in the terminal field
    g, gt = ctx.adjoint_terminal(s, lam), ctx.adjoint_terminal(s, lam * TINY)
    # the forward model is linear in a control this small, and in the larger one
    small = s * 2.0**-500
    w, obs = [t * 2.0**500 for t in ctx.forward(small)]
    wt, obst = ctx.forward(s * TINY)
    ctx.close()
    assert rel(gt, g) < TOL
    assert rel(wt, w) < TOL
    assert rel(obst, obs) < TOL


@pytest.mark.parametrize("n", [16, 64, 256])
def test_subnormal_entries_beside_normal_ones(api, n):
    """One row just above the smallest normal double, the others below it."""
    ctx = api.Context(api.Config(n=n, nsteps=1, dt=1e-3, nu=1e-3, px=1, every=1, store=False))
    s = cu(synthetic.random_field(n, 5)[None])
    s[0, 1::2] *= 0.125
    lift = 2.0 / float(s.abs().max())  # the largest entry is 2^-1021
    w = ctx.omega_from_control(s * lift)
    wt = ctx.omega_from_control(s * lift * 2.0**-1022)
    ctx.close()
    a, b = torch.view_as_real(wt) * 2.0**600 * 2.0**422, torch.view_as_real(w)
    assert float(torch.linalg.norm(a - b) / torch.linalg.norm(b)) < 2.0**-40
