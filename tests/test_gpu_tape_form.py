"""A kept window tape is read by kernels that lay its records out as the forward did:
after a change of team size or specialisation that changes the records the taped adjoint
is refused, after one that does not it returns the same gradients."""
import numpy as np
import pytest

from paper_2204_07137_gb300 import inputs as I
from test_gpu_tape import _inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2204_07137_gb300 import build
    build.build()


def _taped(h):
    from paper_2204_07137_gb300.sim import Simulator
    groups = [(I.ant(), 13)]
    sim = Simulator(groups, form="batched", h_max=h)
    sim.set_window_tape(True)
    return sim, _inputs(sim, groups, h, seed=4)


CHANGES = [("narrower than the lane form", lambda s: s.set_launch(0, 8, 0), lambda s: s.set_launch(0, 16, 0)),
           ("specialised", lambda s: s.specialize(), lambda s: s.specialize(False))]


@pytest.mark.parametrize("what,change,back", CHANGES)
def test_records_of_another_form_are_refused(what, change, back):
    from paper_2204_07137_gb300 import _lib
    h = 3
    sim, (q0, qd0, act, rb, qtb, qdtb) = _taped(h)
    f = sim.window_forward(q0, qd0, act)
    ref = sim.window_adjoint(f[0], f[1], act, rb, qtb, qdtb)
    change(sim)
    with pytest.raises(_lib.ShacError) as e:
        sim.window_adjoint(f[0], f[1], act, rb, qtb, qdtb)
    assert e.value.status == 1      # SHAC_ERR_INVALID_ARG
    sim.step_adjoint(q0, qd0, act[0], qtb[1], qdtb[1], rb[0])    # steps keep no tape
    back(sim)
    got = sim.window_adjoint(f[0], f[1], act, rb, qtb, qdtb)
    change(sim)                      # a forward of the new form goes with it
    f = sim.window_forward(q0, qd0, act)
    new = sim.window_adjoint(f[0], f[1], act, rb, qtb, qdtb)
    torch.cuda.synchronize()
    for x, y, z in zip(ref, got, new):
        assert torch.equal(x, y)
        np.testing.assert_allclose(x.cpu().numpy(), z.cpu().numpy(), rtol=1e-3, atol=1e-3 * float(x.abs().max()))


def test_records_of_the_same_form_are_read():
    h = 3
    sim, (q0, qd0, act, rb, qtb, qdtb) = _taped(h)
    f = sim.window_forward(q0, qd0, act)
    ref = sim.window_adjoint(f[0], f[1], act, rb, qtb, qdtb)
    sim.set_launch(0, 32, 2)
    got = sim.window_adjoint(f[0], f[1], act, rb, qtb, qdtb)
    torch.cuda.synchronize()
    for x, y in zip(ref, got):
        assert torch.equal(x, y)


def test_the_search_for_a_launch_shape_keeps_the_tape():
    """Its timed windows keep their tapes in a workspace of their own; afterwards the
    caller's tape is read if the shape found has its records, refused if not."""
    from paper_2204_07137_gb300 import _lib
    h = 2
    sim, (q0, qd0, act, rb, qtb, qdtb) = _taped(h)
    f = sim.window_forward(q0, qd0, act)
    ref = sim.window_adjoint(f[0], f[1], act, rb, qtb, qdtb)
    sim.autotune_native(budget_ms=200)
    if sim.get_launch(0)[0] >= 16:
        got = sim.window_adjoint(f[0], f[1], act, rb, qtb, qdtb)
        torch.cuda.synchronize()
        for x, y in zip(ref, got):
            assert torch.equal(x, y)
    sim.set_launch(0, 8, 0)
    with pytest.raises(_lib.ShacError) as e:
        sim.window_adjoint(f[0], f[1], act, rb, qtb, qdtb)
    assert e.value.status == 1
    assert sim.status() == 0
