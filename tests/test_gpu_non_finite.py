"""A NaN or an infinity in a member's control, in its trajectory or in one mode
of its terminal adjoint field reaches every mode that depends on it -- the
final state, the adjoint at the window's start, the shell spectra of the
member and of the ensemble mean -- and no bit of another member."""
import numpy as np
import pytest

from paper_2602_14016_gb300 import synthetic

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

NAN, INF = float("nan"), float("inf")


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.fail("a GPU test ran without a GPU")
    from paper_2602_14016_gb300 import api as A, build

    build.build()
    return A


def cu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def results(ctx, s, lam):
    member, mean = ctx.adjoint_spectra(s, lam, 1)
    lam0, filtered = ctx.last_adjoint()
    w, obs = ctx.forward(s)
    return {k: t.clone() for k, t in dict(member=member, mean=mean, lam0=lam0, filtered=filtered, w=w, obs=obs,
                                          grad=ctx.adjoint_terminal(s, lam)).items()}


# bad control, a control whose squares overflow, a bad ordinary mode of the
# terminal field, its mean mode, and a bad control against no adjoint at all
WHERE = [("control", NAN), ("control", -INF), ("blown", 1e160), ("mode", NAN), ("mode", INF), ("mean", NAN),
         ("mean", INF), ("zero_adjoint", NAN)]


@pytest.mark.parametrize("n", [16, 64, 256])
@pytest.mark.parametrize("plain", [False, True])
@pytest.mark.parametrize("where,bad", WHERE)
def test_non_finite_input_reaches_all_that_depends_on_it(api, n, plain, where, bad):
    ctx = api.Context(api.Config(n=n, nsteps=2, dt=1e-3, nu=1e-3, px=4, every=1,
                                 kernels=[api.KernelSpec("exp_abs", 0.2)] * 2))
    if plain:
        ctx.time_kernels("adj_cols")  # the plain sequence of pass kernels
    s = ctx.control_from_omega(cu(np.stack([synthetic.random_vorticity_hat(n, 3 + b) for b in range(2)])))
    lam = cu(np.stack([synthetic.unit_norm_terminal_hat(n, 5 + b) for b in range(2)]))
    want = results(ctx, s, lam)
    kept = cu(synthetic.retained_mask(n))
    some = want["member"][0] > 0  # shells that hold a mode
    s, lam = s.clone(), lam.clone()
    if where in ("control", "zero_adjoint"):
        s[0, n // 3, 1] = bad
    if where == "zero_adjoint":
        lam[0] = 0
    if where == "blown":
        s[0] *= bad
    if where in ("mode", "mean"):
        i, j = (3, 2) if where == "mode" else (0, 0)
        lam[0, i, j] = torch.complex(torch.tensor(bad, dtype=torch.float64), torch.tensor(0.0, dtype=torch.float64))
    got = results(ctx, s, lam)
    ctx.close()
    for k in ("lam0", "filtered", "w", "obs", "grad", "member"):
        assert torch.equal(got[k][1], want[k][1]), k
    assert not torch.isfinite(got["lam0"][0][kept]).any()
    assert not torch.isfinite(got["filtered"][0]).any() and not torch.isfinite(got["grad"][0]).any()
    # slot 0 is the terminal field itself
    assert not torch.isfinite(got["member"][0, 1:][some[1:]]).any()
    assert not torch.isfinite(got["mean"][1:][some[1:]]).any()
    if where in ("control", "zero_adjoint", "blown"):
        assert not torch.isfinite(got["w"][0][kept]).any() and not torch.isfinite(got["obs"][0]).any()
        assert torch.equal(got["member"][0, 0], want["member"][0, 0]) or where == "zero_adjoint"
    else:
        assert torch.equal(got["w"], want["w"]) and torch.equal(got["obs"], want["obs"])
