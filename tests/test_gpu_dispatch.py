"""Every route of an evaluation gives the same bits: whole windows in one
kernel and batches in parts on side streams against the plain sequence of pass
kernels on one stream (which runs while a kernel class is timed), launched
directly, replayed as a graph and captured by the caller."""
import numpy as np
import pytest

from paper_2602_14016_gb300 import synthetic

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.fail("a GPU test ran without a GPU")
    from paper_2602_14016_gb300 import api as A, build

    build.build()
    return A


def make(api, n, plan, B, nsteps, every, ckpt=0, forced=False, t0=False, px=4):
    cfg = api.Config(n=n, nsteps=nsteps, dt=0.3 / n, nu=1e-3, px=px, every=every, include_t0=t0, ckpt_every=ckpt,
                     forcing="kolmogorov" if forced else "none",
                     kernels=[api.KernelSpec("exp_abs", 0.1 * (b % 4)) for b in range(B)])
    ctx = api.Context(cfg)
    ctx.set_plan(plan)
    s = ctx.control_from_omega(torch.from_numpy(np.stack([synthetic.random_vorticity_hat(n, b) for b in range(B)])).cuda())
    gen = torch.Generator("cuda").manual_seed(n + B)
    ctx.set_observations(torch.randn((B, ctx.nt, px * px, 2), dtype=torch.float64, device="cuda", generator=gen))
    lam = torch.from_numpy(np.stack([synthetic.unit_norm_terminal_hat(n, 50 + b) for b in range(B)])).cuda()
    return ctx, s, lam


def results(ctx, s, lam, spectra=True):
    J, g = ctx.cost_grad(s)
    out = [J.clone(), g.clone()]
    w, o = ctx.forward(s)
    out += [w.clone(), o.clone(), ctx.vjp(o, w).clone(), ctx.adjoint_terminal(s, lam).clone()]
    if spectra:
        out += [t.clone() for t in ctx.adjoint_spectra(s, lam, 1)]
    return out


def same(a, b):
    return all(torch.equal(x, y) for x, y in zip(a, b)) and len(a) == len(b)


# windows up to and beyond the batch at which they run in one kernel; batches
# on both sides of the line from which they run in parts, and of the number of parts
WINDOWS = [(16, 0, 1), (16, 0, 5), (32, 0, 3), (32, 1, 128), (32, 1, 129), (64, 0, 16), (64, 0, 17), (64, 1, 4), (64, 1, 5),
           (64, 2, 2)]
PARTS = [(128, 3, 9), (128, 3, 10), (256, 0, 4), (256, 0, 5), (256, 1, 10), (512, 0, 3), (1024, 2, 2)]


@pytest.mark.parametrize("n,plan,B", WINDOWS + PARTS)
@pytest.mark.parametrize("ckpt,forced,t0", [(0, False, True), (2, True, False)])
def test_routes_agree_bitwise(api, n, plan, B, ckpt, forced, t0):
    ctx, s, lam = make(api, n, plan, B, 3, 1, ckpt, forced, t0)
    got = results(ctx, s, lam)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        again = results(ctx, s, lam)
    torch.cuda.current_stream().wait_stream(side)
    ctx.set_graphs(True)
    replayed = results(ctx, s, lam)
    ctx.set_graphs(False)
    w, o = ctx.forward(s)
    ctx.time_kernels("fwd_rows")
    crossed = ctx.vjp(o, w)  # the passes read what the other route stored
    plain = results(ctx, s, lam)
    ctx.close()
    assert torch.count_nonzero(plain[1]) > 0
    assert same(got, plain) and same(again, plain) and same(replayed, plain) and torch.equal(crossed, plain[4])


@pytest.mark.parametrize("n,plan,B", [(32, 0, 3), (64, 0, 2), (256, 0, 5)])
def test_members_of_their_own_windows_agree_bitwise(api, n, plan, B):
    ctx, s, _ = make(api, n, plan, B, 4, 2, forced=True)
    for b in range(B):
        ctx.set_member(b, nsteps=4 if b % 2 == 0 else 2, px=4 >> (b % 2), nu=1e-3 * (1 + b), forcing=b % 2 == 0,
                       kernel=api.KernelSpec("exp_abs", 0.2),
                       m=torch.full(((2 if b % 2 == 0 else 1), (4 >> (b % 2)) ** 2, 2), 0.1 * b, dtype=torch.float64, device="cuda"))
    a = [t.clone() for t in ctx.cost_grad(s)]
    ctx.time_kernels("adj_cols")
    b = [t.clone() for t in ctx.cost_grad(s)]
    ctx.close()
    assert same(a, b)


@pytest.mark.parametrize("n,plan,B", [(32, 0, 3), (64, 2, 1), (256, 0, 5), (512, 0, 3)])
def test_caller_captures_an_evaluation(api, n, plan, B):
    ctx, s, _ = make(api, n, plan, B, 2, 1)
    want = [t.clone() for t in ctx.cost_grad(s)]
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        out = ctx.cost_grad(s)
    for t in out:
        t.zero_()
    graph.replay()
    torch.cuda.synchronize()
    got = [t.clone() for t in out]
    ctx.close()
    assert same(got, want)


# batches on both sides of the line up to which column passes load their inputs early
@pytest.mark.parametrize("n,plan,few,many", [(256, 0, 3, 4), (256, 1, 7, 8), (512, 0, 1, 2), (512, 2, 3, 4)])
def test_members_do_not_depend_on_their_batch(api, n, plan, few, many):
    out = []
    for B in (few, many):
        ctx, s, lam = make(api, n, plan, B, 2, 1, forced=True)
        ctx.set_observations(torch.full((B, ctx.nt, 16, 2), 0.25, dtype=torch.float64, device="cuda"))
        out.append([t[:few].clone() for t in results(ctx, s, lam, spectra=False)])
        ctx.close()
    assert same(*out)
