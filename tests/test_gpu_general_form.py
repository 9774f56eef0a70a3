"""The general kernels on the models at the edges of the lane form: a second group with
more links than a team has lanes takes the whole batch to the general kernels, whatever
the team size.  Step and step adjoint against the FP64 oracle."""
import numpy as np
import pytest

from helpers import assert_grad_close, assert_state_close, oracle_step_with_floor
from paper_2204_07137_gb300 import inputs as I
from test_gpu_form_rounding import T, many_links
from test_gpu_lane_form import MODELS

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2204_07137_gb300 import build
    build.build()


@pytest.mark.parametrize("name", MODELS)
def test_general_kernels_match_oracle(oracle_mod, name):
    from paper_2204_07137_gb300.sim import Simulator
    m, N = MODELS[name](), 11
    o = oracle_mod.Oracle(m)
    q, qd = I.random_state(m, N, 4, pos_scale=0.2, vel_scale=0.5)
    if name == "body":
        q[2] = np.float32(m.root_z)
    a = I.window_actions(m, N, 1, 4)[0]
    rng = np.random.default_rng(5)
    bars = [rng.normal(size=x).astype(np.float32) for x in ((m.nq, N), (m.nv, N), (N,))]
    (rq, rqd, rr), (fq, fqd, fr) = oracle_step_with_floor(o, q.T, qd.T, a.T)
    ref = np.concatenate([x.T for x in o.step_vjp(q.T, qd.T, a.T, bars[0].T, bars[1].T, bars[2])])
    one = lambda x: torch.cat([T(x), torch.zeros(1, device="cuda")])  # noqa: E731   the other group's environment
    sim = Simulator([(m, N), (many_links(), 1)], form="batched", h_max=1)
    for lanes in (0, 4, 32):
        sim.set_launch(0, lanes, 0)
        tag = f"{name}/general/T{sim.get_launch(0)[0]}"
        out = sim.step(one(q), one(qd), one(a))
        g = sim.step_adjoint(one(q), one(qd), one(a), *(one(x) for x in bars))
        torch.cuda.synchronize()
        assert sim.status() == 0
        qn, qdn, gq, gqd, ga = (x.cpu().numpy()[:k * N].reshape(k, N)
                                for x, k in zip((*out[:2], *g), (m.nq, m.nv, m.nq, m.nv, m.na)))
        assert_state_close(qn.T, rq, f"{tag} q", fq)
        assert_state_close(qdn.T, rqd, f"{tag} qd", fqd)
        assert_state_close(out[2].cpu().numpy()[:N], rr, f"{tag} reward", fr)
        assert_grad_close(np.concatenate([gq, gqd, ga]), ref, f"{tag} step adjoint")


def test_batches_take_the_form_they_should():
    """Seen from outside in the 152-muscle model's scratch: 36 KB an environment in lane
    form, 60 KB in general, so a CTA holds more warps."""
    from paper_2204_07137_gb300.sim import Simulator
    warps = []
    for groups in ([(I.mtu(), 4)], [(I.mtu(), 4), (many_links(), 1)]):
        sim = Simulator(groups, form="batched", h_max=1)
        sim.set_launch(-1, 0, 8)
        warps.append(sim.get_launch(0)[1])
    assert warps[0] > warps[1], warps
