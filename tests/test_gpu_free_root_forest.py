"""A free root beside a second tree fixed to the world, both with contacts.  Only the
free root's tree has its positions relative to the root origin, so only its contacts
add the root height to their depth (and give their depth's cotangent to it): step and
step adjoint against the FP64 oracle in every form."""
import numpy as np
import pytest

from helpers import assert_grad_close, assert_state_close, oracle_step_with_floor
from paper_2204_07137_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2204_07137_gb300 import build
    build.build()


def T(x):
    return torch.from_numpy(np.ascontiguousarray(np.asarray(x, np.float32).reshape(-1))).cuda()


def body_and_arm():
    b = I._Builder("body and arm")
    m, c, J = I.capsule_mass_inertia(0.1, (0, 0, 0), (0.1, 0, 0.2), 500.0)
    root = b.link(-1, I.FREE, mass=m, com=c, inertia=J)
    leg = b.link(root, I.REVOLUTE, axis=(0, 1, 0), pos=(0, 0, -0.2), mass=0.5, com=(0, 0, -0.1), inertia=0.01 * np.eye(3))
    arm = b.link(-1, I.REVOLUTE, axis=(0, 1, 0), pos=(1.0, 0, 0.5), mass=0.7, com=(0, 0, -0.2), inertia=0.02 * np.eye(3))
    tip = b.link(arm, I.FIXED, pos=(0, 0, -0.45), mass=0.2, com=(0, 0, 0), inertia=0.001 * np.eye(3))
    b.contact(leg, (0, 0, -0.2), 0.06)
    b.contact(tip, (0, 0, 0), 0.06)
    return b.finish(act_dof=[6, 7], act_gear=[5.0, 5.0], dt=I.CONTROL_DT, substeps=4, ke=2e3, kd=50.0, kt=50.0, mu=0.5,
                    armature=0.05, damping=0.1, root_z=0.45)


@pytest.mark.parametrize("form,lanes,spec", [("plain", 0, False), ("batched", 8, False), ("batched", 16, False),
                                             ("batched", 16, True)])
def test_step_and_adjoint_match_oracle(oracle_mod, form, lanes, spec):
    from paper_2204_07137_gb300.sim import Simulator
    m, N = body_and_arm(), 37
    sim = Simulator([(m, N)], form=form, h_max=1)
    if lanes:
        sim.set_launch(0, lanes, 0)      # 9 lanes needed: 8 run the general kernels
    if spec:
        sim.specialize()
    o = oracle_mod.Oracle(m)
    q, qd = I.initial_state(m, N, 3)
    a = I.window_actions(m, N, 1, 3)[0]
    rng = np.random.default_rng(5)
    bars = [rng.normal(size=x).astype(np.float32) for x in ((m.nq, N), (m.nv, N), (N,))]
    (rq, rqd, rr), (fq, fqd, fr) = oracle_step_with_floor(o, q.T, qd.T, a.T)
    ref = np.concatenate([x.T for x in o.step_vjp(q.T, qd.T, a.T, bars[0].T, bars[1].T, bars[2])])
    qn, qdn, r = sim.step(T(q), T(qd), T(a))
    g = sim.step_adjoint(T(q), T(qd), T(a), *(T(x) for x in bars))
    torch.cuda.synchronize()
    tag = f"body and arm/{form}/T{lanes}{'/spec' if spec else ''}"
    assert_state_close(qn.cpu().numpy().reshape(m.nq, N).T, rq, f"{tag} q", fq)
    assert_state_close(qdn.cpu().numpy().reshape(m.nv, N).T, rqd, f"{tag} qd", fqd)
    assert_state_close(r.cpu().numpy(), rr, f"{tag} reward", fr)
    got = np.concatenate([x.cpu().numpy().reshape(-1, N) for x in g])
    assert_grad_close(got, ref, f"{tag} step adjoint")
