"""The lane form of the batched kernels (a lane per link and DOF) at the edges of
its range: one link, one hinge, links without a DOF on the lanes after the DOFs,
the deepest tree a team can hold, muscles whose items crowd on two links, and a
muscle too few for the form's records (the general kernels take that batch).
Step and step adjoint against the FP64 oracle at the repository's tolerances,
generic and model-specialised, at the default team size and at a narrower one
that takes the general kernels."""
import numpy as np
import pytest

from helpers import assert_grad_close, assert_state_close, long_chain, oracle_step_with_floor
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


def _finish(b, n_act, **kw):
    return b.finish(act_dof=list(range(n_act)), act_gear=[5.0] * n_act, dt=I.CONTROL_DT, substeps=4, armature=0.05,
                    damping=0.1, **kw)


def one_hinge():
    b = I._Builder("hinge")
    b.link(-1, I.REVOLUTE, axis=(0, 1, 0), mass=0.5, com=(0, 0, -0.3), inertia=np.diag([0.02, 0.02, 0.001]),
           limit=(-0.1, 0.1))
    return _finish(b, 1, k_limit=100.0, rw_q=[0.1])


def free_body():
    b = I._Builder("body")
    m, c, J = I.capsule_mass_inertia(0.1, (0, 0, 0), (0.1, 0, 0.2), 500.0)
    root = b.link(-1, I.FREE, mass=m, com=c, inertia=J)
    b.contact(root, (0, 0, 0), 0.1)
    return b.finish(act_dof=[0, 4], act_gear=[0.1, 5.0], dt=I.CONTROL_DT, substeps=4, ke=5e3, kd=100.0, kt=50.0, mu=0.5,
                    damping=0.1, root_z=0.099)


def fixed_tail():
    """Two hinges, then five links without a DOF."""
    b = I._Builder("tail")
    m, c, J = I.capsule_mass_inertia(0.03, (0, 0, 0), (0, 0, -0.2), 1000.0)
    k = b.link(-1, I.REVOLUTE, axis=(0, 1, 0), mass=m, com=c, inertia=J)
    k = b.link(k, I.REVOLUTE, axis=(1, 0, 0), pos=(0, 0, -0.2), mass=m, com=c, inertia=J)
    for j in range(5):
        k = b.link(k, I.FIXED, pos=(0.02 * j, 0, -0.1), quat=(0, 0, 0.1, 0.995), mass=0.1, com=(0, 0.01, 0),
                   inertia=np.diag([1e-4, 1e-4, 1e-4]))
    return _finish(b, 2)


def muscled(n):
    """Four hinges and n muscles, nearly all between the first two links."""
    rng = np.random.default_rng(n)
    b = I._Builder("muscled")
    m, c, J = I.capsule_mass_inertia(0.04, (0, 0, 0), (0, 0, -0.3), 1000.0)
    links = [b.link(-1, I.REVOLUTE, axis=(0, 1, 0), mass=m, com=c, inertia=J)]
    for j in range(3):
        links.append(b.link(links[-1], I.REVOLUTE, axis=(0, 1, 0) if j % 2 else (1, 0, 0), pos=(0, 0, -0.3), mass=m, com=c,
                            inertia=J))
    for k in range(n):
        pair = (links[0], links[1]) if k % 8 else (links[2], links[3])
        b.muscle(float(rng.uniform(20.0, 60.0)),
                 [(lk, rng.uniform(-0.05, 0.05, 3) + np.array([0, 0, -0.15])) for lk in pair])
    return b.finish(act_dof=[], act_gear=[], dt=I.CONTROL_DT, substeps=4, armature=0.05, damping=0.5)


MODELS = {"hinge": one_hinge, "body": free_body, "tail": fixed_tail, "chain32": lambda: long_chain(26),
          "muscles 1": lambda: muscled(1), "muscles 45": lambda: muscled(45)}


@pytest.mark.parametrize("spec", [False, True])
@pytest.mark.parametrize("name", MODELS)
def test_lane_form_edges_match_oracle(oracle_mod, name, spec):
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
    for narrow in (False, True):
        sim = Simulator([(m, N)], form="batched", h_max=1)
        lanes = sim.get_launch(0)[0]
        if narrow:
            sim.set_launch(0, max(1, lanes // 2), 0)
        if spec:
            sim.specialize()
        tag = f"{name}{'/spec' if spec else ''}/T{sim.get_launch(0)[0]}"
        qn, qdn, r = sim.step(T(q), T(qd), T(a))
        g = sim.step_adjoint(T(q), T(qd), T(a), *(T(x) for x in bars))
        torch.cuda.synchronize()
        assert sim.status() == 0
        assert_state_close(qn.cpu().numpy().reshape(m.nq, N).T, rq, f"{tag} q", fq)
        assert_state_close(qdn.cpu().numpy().reshape(m.nv, N).T, rqd, f"{tag} qd", fqd)
        assert_state_close(r.cpu().numpy(), rr, f"{tag} reward", fr)
        got = np.concatenate([g[0].cpu().numpy().reshape(m.nq, N), g[1].cpu().numpy().reshape(m.nv, N),
                              g[2].cpu().numpy().reshape(m.na, N)])
        assert_grad_close(got, ref, f"{tag} step adjoint")
