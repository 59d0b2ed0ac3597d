"""What a co-batching run reports of its members: those that ran together."""
import numpy as np
import pytest

from paper_2602_14016_gb300 import serve, synthetic

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def jobs(arrivals):
    out = []
    for i, t in enumerate(arrivals):
        s0 = synthetic.random_field(32, 10 + i)
        out.append(serve.Job(job_id=i, n=32, nsteps=10, dt=5e-3, nu=1e-3, px=4, every=5, kernel=("exp_abs", 0.5), iters=2,
                             arrival=t, m=np.zeros((1, 2, 16, 2)), s0=s0[None].copy()))
    return out


def test_members_that_never_ran_together_are_not_counted_together():
    srv = serve.CoBatchServer({32: dict(slots=3, nsteps=10, px=4, dt=5e-3)}, every=5)
    srv.run(jobs([0.0]))  # kernels are loaded, a slot has been used
    apart = srv.run(jobs([0.0, 3.0]))
    assert apart["failed"] == 0 and apart["peak_running"] == 1 and apart["peak_members"] >= 2
    together = srv.run(jobs([0.0, 0.0, 0.0]))
    assert together["failed"] == 0 and together["peak_running"] == 3
    srv.close()
