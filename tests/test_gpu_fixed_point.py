"""The block fixed-point transforms of the pass kernels at the edges of their
range: powers of two of the adjoint field (every exponent moves with it),
states whose columns differ by hundreds of orders of magnitude or vanish,
single modes, impulses, and non-finite states."""
import numpy as np
import pytest

from cases import make_pair
from conftest import rel
from paper_2602_14016_gb300 import synthetic

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SIZES = [16, 32, 64, 128, 256, 512, 1024]
# A few steps on unit fields leave at most a few hundred roundings of 2^-53,
# amplified by the derivatives only in the highest modes: 1e-12 of the norm,
# the step tolerance of the parity tests.
TOL = 1e-12


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.fail("a GPU test ran without a GPU")
    from paper_2602_14016_gb300 import api as A, build

    build.build()
    return A


def cu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("n", SIZES)
def test_adjoint_scales_exactly_by_powers_of_two(api, n):
    """The adjoint is linear in the terminal field, and a power of two changes
    exponents only: the gradient is bitwise the scaled one, far outside the
    ordinary range of magnitudes too."""
    for v in range(api.N.load().da_plan_count(n)):
        ctx = api.Context(api.Config(n=n, nsteps=2, dt=1e-3, nu=1e-3, px=1, every=2))
        ctx.set_plan(v)
        s = ctx.control_from_omega(cu(synthetic.random_vorticity_hat(n, 3)[None]))
        lam = cu(synthetic.unit_norm_terminal_hat(n, 4)[None])
        g = ctx.adjoint_terminal(s, lam)
        assert torch.count_nonzero(g) > 0
        for k in (-700, -300, 300, 700):
            assert torch.equal(ctx.adjoint_terminal(s, lam * 2.0**k), g * 2.0**k)
        ctx.close()


def states(n):
    K = (n - 1) // 3
    _, KY = synthetic.wavenumbers(n)
    w = synthetic.random_vorticity_hat(n, 8)
    tiny = w.copy()
    tiny[:, 1::2] *= 1e-200  # every other column all but gone
    one = np.zeros_like(w)
    one[K, K] = n * n / 2.0  # the corner of the retained set
    column = np.where(np.arange(n // 2 + 1)[None, :] == 0, w, 0)  # kx = 0 only: v = 0
    impulse = np.where(synthetic.retained_mask(n), np.exp(-1j * KY * 2 * np.pi * 3 / n), 0)
    impulse[0, 0] = 0
    return {"columns": tiny, "corner": one, "kx0": column, "impulse": impulse * 0.1}


@pytest.mark.parametrize("n", [16, 64, 256])
@pytest.mark.parametrize("name", ["columns", "corner", "kx0", "impulse"])
def test_uneven_states_match_the_oracle(orc, api, n, name):
    probs, cfg = make_pair(orc, n, 2, 1e-3, 1e-3, px=8, every=1)
    P = probs[0]
    w = states(n)[name]
    for v in range(api.N.load().da_plan_count(n)):
        ctx = api.Context(cfg)
        ctx.set_plan(v)
        s = orc.control_from_omega(P, w)
        wT, obs = ctx.forward(cu(s[None]))
        rw, robs = orc.forward(P, s)
        assert rel(wT.cpu().numpy()[0], rw) < TOL
        assert np.abs(obs.cpu().numpy()[0] - robs).max() <= TOL * np.abs(robs).max()
        m = np.zeros_like(robs)
        J, g, _ = orc.cost_grad(P, s, m)
        ctx.set_observations(cu(m[None]))
        Jg, gg = ctx.cost_grad(cu(s[None]))
        assert abs(Jg.item() - J) <= TOL * J
        assert rel(gg.cpu().numpy()[0], g) < TOL
        ctx.close()


@pytest.mark.parametrize("n", [16, 64, 512])
@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf")])
def test_non_finite_members_stay_their_own(api, n, bad):
    """A NaN or an infinity in one member's control makes that member's cost
    and gradient non-finite and leaves the other member's bits alone."""
    cfg = api.Config(n=n, nsteps=2, dt=1e-3, nu=1e-3, px=4, every=1, kernels=[api.KernelSpec("exp_abs", 0.2)] * 2)
    ctx = api.Context(cfg)
    s = ctx.control_from_omega(cu(np.stack([synthetic.random_vorticity_hat(n, 3 + b) for b in range(2)])))
    ctx.set_observations(torch.zeros((2, 2, 16, 2), dtype=torch.float64, device="cuda"))
    J, g = ctx.cost_grad(s)
    s2 = s.clone()
    s2[0, n // 3, 1] = bad
    J2, g2 = ctx.cost_grad(s2)
    assert not torch.isfinite(J2[0]) and not torch.isfinite(g2[0]).any()
    assert torch.equal(J2[1], J[1]) and torch.equal(g2[1], g[1])
