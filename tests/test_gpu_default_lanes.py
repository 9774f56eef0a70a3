"""Default team sizes: a lane for every DOF and every link without one, whatever the
batch size, so that a model takes the same kernels in every batch and a window over
environment ranges equals one over all of them, bit for bit."""
import numpy as np
import pytest

from helpers import assert_grad_close, assert_state_close, oracle_step_with_floor
from paper_2204_07137_gb300 import inputs as I
from test_gpu_form_rounding import T
from test_gpu_lane_form import muscled

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2204_07137_gb300 import build
    build.build()


def free_with(hinges, fixed):
    """A free root with hinges and links without a DOF on it, a contact on the root."""
    b = I._Builder(f"free {hinges} {fixed}")
    J = np.diag([0.01, 0.012, 0.008])
    root = b.link(-1, I.FREE, mass=2.0, com=(0, 0, 0.05), inertia=4 * J)
    for k in range(hinges):
        b.link(root, I.REVOLUTE, axis=(0, 1, 0) if k % 2 else (1, 0, 0), pos=(0.1 * k, 0.05, -0.1), mass=0.3,
               com=(0.01, 0, -0.1), inertia=J)
    for k in range(fixed):
        b.link(root, I.FIXED, pos=(0, 0.1 * k, 0.1), quat=(0, 0.1, 0, 0.995), mass=0.1, com=(0, 0.02, 0), inertia=0.1 * J)
    b.contact(root, (0, 0, 0), 0.15)
    return b.finish(act_dof=[6], act_gear=[2.0], dt=I.CONTROL_DT, substeps=4, armature=0.05, damping=0.1, ke=2e3, kd=50.0,
                    kt=50.0, mu=0.5, root_z=0.149)


def _window(m, q, qd, act):
    from paper_2204_07137_gb300.sim import Simulator
    N, h = q.shape[1], len(act)
    sim = Simulator([(m, N)], form="batched", h_max=h)
    a = T(act).view(h, -1)
    f = sim.window_forward(T(q), T(qd), a)
    g = sim.window_adjoint(f[0], f[1], a, torch.ones(h, N, device="cuda"), torch.zeros_like(f[0]), torch.ones_like(f[1]))
    torch.cuda.synchronize()
    assert sim.status() == 0
    return sim.get_launch(0)[0], [x.cpu().numpy().reshape(-1, N) for x in (*f, *g)]


# (model, lanes its default team has at least, environments): 8 hinges and 3 fixed links
# need 17 lanes with 14 DOFs and 12 links; 2 hinges and a fixed link need 9 with 8 DOFs.
# The batches are too large for a wider team than that, their halves are not.  Four
# muscles have no lane form.
@pytest.mark.parametrize("make,need,N", [(lambda: free_with(8, 3), 17, 11), (lambda: free_with(2, 1), 9, 2600),
                                         (lambda: muscled(4), 4, 9000)])
def test_kernels_do_not_depend_on_the_batch_size(oracle_mod, make, need, N):
    m = make()
    q, qd = I.initial_state(m, N, 4)
    qd = (qd + np.random.default_rng(4).uniform(-0.3, 0.3, qd.shape)).astype(np.float32)
    act = I.window_actions(m, N, 2, 4)
    lanes, whole = _window(m, q, qd, act)
    assert lanes >= need
    k = N // 2
    _, lo = _window(m, q[:, :k], qd[:, :k], act[:, :, :k])
    _, hi = _window(m, q[:, k:], qd[:, k:], act[:, :, k:])
    for w, a, b in zip(whole, lo, hi):
        np.testing.assert_array_equal(w, np.concatenate([a, b], 1))
    # the first step of some environments against the oracle
    o, n = oracle_mod.Oracle(m), 11
    (rq, rqd, _), (fq, fqd, _) = oracle_step_with_floor(o, q[:, :n].T, qd[:, :n].T, act[0, :, :n].T)
    assert_state_close(whole[0].reshape(3, m.nq, N)[1, :, :n].T, rq, f"{m.name} q", fq)
    assert_state_close(whole[1].reshape(3, m.nv, N)[1, :, :n].T, rqd, f"{m.name} qd", fqd)


def test_groups_share_the_gpu():
    """Groups widen together only while all their warps fit at once."""
    from paper_2204_07137_gb300.sim import Simulator
    m = I.cartpole()
    alone = Simulator([(m, 1024)], form="batched", h_max=1).get_launch(0)[0]
    assert alone == 16
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    sim = Simulator([(m, 1024), (I.ant(), 16 * sms)], form="batched", h_max=1)
    assert sim.get_launch(1)[0] == 16 and sim.get_launch(0)[0] == 2
    sim.set_launch(0, 8, 0)
    sim.set_launch(0, 0, 0)
    assert sim.get_launch(0)[0] == 2
