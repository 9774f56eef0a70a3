"""The lane form's generic kernels round as the general kernels: a model without
muscles has the same states, to the last bit, whichever of the two its batch takes,
so contact, friction and limit switches fall the same way and the window gradients,
which jump there, agree.  The general kernels are made to run by a second group that
has more links than a team has lanes (a batch takes the lane form only as a whole)."""
import numpy as np
import pytest

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


def skewed_tree():
    """Free root, a prismatic joint and hinges about general axes, full inertias,
    two branches and a link without a DOF."""
    J = np.array([[2.0, 0.3, 0.1], [0.3, 1.5, -0.2], [0.1, -0.2, 1.1]])
    b = I._Builder("skewed")
    root = b.link(-1, I.FREE, mass=3.0, com=(0.1, 0.2, -0.1), inertia=0.1 * J)
    k = b.link(root, I.REVOLUTE, axis=(1, 0.3, 0), pos=(0.1, 0.05, -0.2), mass=0.5, com=(0.02, 0.03, 0.1), inertia=0.01 * J,
               limit=(-0.05, 0.05))
    b.link(k, I.PRISMATIC, axis=(0.2, 0.1, 1), pos=(0, 0.1, -0.1), mass=0.4, com=(0, 0.02, 0.05), inertia=0.01 * J)
    k = b.link(root, I.FIXED, pos=(-0.1, 0, 0), quat=(0, 0.1, 0, 0.995), mass=0.2, com=(0.01, 0, 0), inertia=0.002 * J)
    foot = b.link(k, I.REVOLUTE, axis=(0, 1, 0.4), pos=(0, 0, -0.2), mass=0.5, com=(0.02, 0.03, 0.1), inertia=0.01 * J)
    for c in (root, foot):
        b.contact(c, (0, 0.02, -0.05), 0.1)
    return b.finish(act_dof=[6, 8], act_gear=[3.0, 2.0], dt=I.CONTROL_DT, substeps=16, armature=0.01, damping=0.1, ke=5e3,
                    kd=100.0, kt=300.0, mu=0.7, k_limit=200.0, root_z=0.25)


def many_links():
    """One hinge and 33 fixed links: more than a team's lanes."""
    b = I._Builder("many")
    k = b.link(-1, I.REVOLUTE, axis=(0, 1, 0), mass=0.5, com=(0, 0, -0.3), inertia=np.diag([0.02, 0.02, 0.001]))
    for _ in range(33):
        k = b.link(k, I.FIXED, pos=(0.01, 0, 0), mass=0.01, com=(0, 0, 0), inertia=np.diag([1e-5] * 3))
    return b.finish(act_dof=[0], act_gear=[1.0], dt=I.CONTROL_DT, substeps=2)


MODELS = {"cartpole": (I.cartpole, 70), "ant": (I.ant, 300), "hopper": (I.hopper, 100), "halfcheetah": (I.halfcheetah, 100),
          "humanoid": (I.humanoid, 60), "skewed": (skewed_tree, 300)}


def _window(m, N, h, seed, lane_form):
    """The group's [k, N] states and gradients of an open-loop window."""
    from paper_2204_07137_gb300.sim import Simulator
    groups = [(m, N)] + ([] if lane_form else [(many_links(), 1)])
    sim = Simulator(groups, form="batched", h_max=h)
    q, qd = I.initial_state(m, N, seed)
    act = I.window_actions(m, N, h, seed)
    pad = lambda x, lead: torch.cat([T(x).view(*lead, -1)] + ([] if lane_form else [torch.zeros(*lead, 1, device="cuda")]), -1)  # noqa: E731
    q, qd, act = pad(q, ()), pad(qd, ()), pad(act, (h,))
    f = sim.window_forward(q, qd, act)
    g = sim.window_adjoint(f[0], f[1], act, torch.ones(h, sim.n_envs, device="cuda"),
                           *(torch.zeros(h + 1, n, device="cuda") for n in (sim.q_size, sim.qd_size)))
    torch.cuda.synchronize()
    assert sim.status() == 0
    out = []
    for x, k in zip((*f[:2], *g), (m.nq, m.nv, m.nq, m.nv, m.na)):
        out.append(x[..., :k * N].reshape(-1, N).cpu().numpy())
    return out


@pytest.mark.parametrize("name", MODELS)
def test_states_do_not_depend_on_the_form(name):
    make, N = MODELS[name]
    a, b = _window(make(), N, 6, 3, True), _window(make(), N, 6, 3, False)
    np.testing.assert_array_equal(a[0], b[0])
    np.testing.assert_array_equal(a[1], b[1])


@pytest.mark.parametrize("seed", [1115, 1329, 2466])
def test_gradients_do_not_depend_on_the_form(seed):
    """Batches of which one environment stands within rounding of a switch: another
    rounding of the states moves its gradient by 8 to 20 %.  With the same states
    the gradients differ by the rounding of the reverse pass (measured up to 1e-4 of
    an environment's gradient)."""
    m, N = I.ant(), 1531
    a, b = (np.concatenate(_window(m, N, 2, seed, form)[2:]).astype(np.float64) for form in (True, False))
    err = np.linalg.norm(a - b, axis=0) / np.linalg.norm(b, axis=0)
    assert err.max() < 1e-3, (int(err.argmax()), float(err.max()))


def sliding_ball(contacts=1):
    b = I._Builder("ball")
    root = b.link(-1, I.FREE, mass=1.0, com=(0, 0, 0), inertia=0.01 * np.eye(3))
    for k in range(contacts):
        b.contact(root, (0, 0, 0), 0.1 if k == contacts - 1 else 0.05 + 0.002 * k)
    return b.finish(act_dof=[4], act_gear=[1.0], dt=I.CONTROL_DT, substeps=1, ke=5e3, kd=100.0, kt=20.0, mu=0.5, root_z=0.099)


@pytest.mark.parametrize("contacts", [1, 16, 17])
@pytest.mark.parametrize("switch", ["slip", "touch"])
def test_reverse_takes_the_contact_branch_of_the_forward(switch, contacts):
    """Balls whose sliding speed (or height) steps through its switch a few units in
    the last place at a time, at 64 depths (speeds), vertical speeds and directions.
    The gradient is the one of the branch the force took: the general kernels', which
    keep the forward's depth and force (their branch differs from the other's by
    h kt / m = 0.3 of a unit cotangent; rounding by less than 1e-5).  A link of 16 contacts
    fills a record's word, one of 17 has the general kernels on both sides."""
    from paper_2204_07137_gb300.sim import Simulator
    m, n, steps = sliding_ball(contacts), 64, 129
    rng = np.random.default_rng(2)
    N = n * steps
    depth = np.repeat(rng.uniform(1e-4, 3e-3, n), steps)
    vz = np.repeat(rng.uniform(-0.5, 0.5, n), steps)
    phi = np.repeat(rng.uniform(0, 2 * np.pi, n), steps)
    ulp = np.tile(np.arange(steps) - steps // 2, n) * 2.0 ** -24
    speed = np.repeat(rng.uniform(0.05, 1.0, n), steps)
    if switch == "slip":   # kt v = mu |fn|
        speed = 0.5 * np.abs((-5e3 + 100 * vz) * depth) / 20 * (1 + 4 * ulp)
    else:
        depth = 0.1 * ulp / 16
    q, qd = np.zeros((7, N)), np.zeros((6, N))
    q[2], q[6] = 0.1 - depth, 1.0
    if switch == "touch":  # the contact's height is the root's less the radius: exact steps about zero
        q[2] = np.float32(0.1) + 0.1 * ulp
    qd[3], qd[4], qd[5] = speed * np.cos(phi), speed * np.sin(phi), vz
    out = []
    for lane_form in (True, False):
        sim = Simulator([(m, N)] + ([] if lane_form else [(many_links(), 1)]), form="batched", h_max=1)
        pad = lambda x: torch.cat([T(x)] + ([] if lane_form else [torch.zeros(1, device="cuda")]))  # noqa: E731
        x = [pad(q), pad(qd), pad(np.zeros((1, N)))]
        y = sim.step(*x)
        g = sim.step_adjoint(*x, torch.zeros_like(y[0]), torch.ones_like(y[1]), torch.zeros_like(y[2]))
        torch.cuda.synchronize()
        out.append([v[:k * N].cpu().numpy().reshape(k, N) for v, k in ((y[0], 7), (y[1], 6), (g[0], 7), (g[1], 6))])
    for a, b in zip(out[0][:2], out[1][:2]):
        np.testing.assert_array_equal(a, b)
    # both branches are taken: the sliding's show in the gradients of the horizontal
    # velocities, the contact's in that of the height
    both = out[1][3][3:5] if switch == "slip" else out[1][2][2:3]
    assert len({tuple(v) for v in np.round(both.T, 1)}) > 1
    for a, b in zip(out[0][2:], out[1][2:]):
        np.testing.assert_allclose(a, b, rtol=1e-3, atol=1e-3 * np.abs(b).max())
