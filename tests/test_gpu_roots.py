"""The lane form's reciprocal square root: its error bound over the floats, and steps
whose roots have the smallest and largest arguments (a mass-matrix pivot and a squared
muscle length below the normal floats, a tangential velocity whose square overflows),
which the general kernels compute too."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2204_07137_gb300 import inputs as I
from test_gpu_form_rounding import T, many_links, sliding_ball

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

KERNEL = """
#include "shac_team.cuh"
__global__ void k(const float* x, float* y, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = shac::rsqrt_refined(x[i]);
}
extern "C" int run(const float* x, float* y, int n) {
  k<<<(n + 255) / 256, 256>>>(x, y, n);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2204_07137_gb300 import build
    build.build()


def test_refined_root_error_bound(tmp_path):
    """All exponents of the positive floats, subnormal ones too, 2048 mantissas each,
    dense around powers of two: |y sqrt(x) - 1| <= 1.5 * 2^-24 (half a unit for the last
    rounding, half for that of x y, and the square of rsqrtf's own error)."""
    from paper_2204_07137_gb300 import build
    src, lib = tmp_path / "root.cu", tmp_path / "root.so"
    src.write_text(KERNEL)
    subprocess.check_call([build.nvcc(), *build.ARCH, *build.FLAGS, "-I", build.CSRC, "-shared", str(src), "-o", str(lib)])
    rng = np.random.default_rng(0)
    mant = np.unique(np.concatenate([rng.integers(0, 1 << 23, 2048), np.arange(64), (1 << 23) - 1 - np.arange(64)]))
    bits = (np.arange(255, dtype=np.uint32)[:, None] << 23 | mant[None].astype(np.uint32)).reshape(-1)
    x = bits[bits > 0].view(np.float32)
    x = np.concatenate([x, np.float32([0.0, np.inf])])
    xd, yd = torch.from_numpy(x).cuda(), torch.empty(len(x), device="cuda")
    torch.cuda.synchronize()
    f = ctypes.CDLL(os.fspath(lib)).run
    f.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int]
    assert f(xd.data_ptr(), yd.data_ptr(), len(x)) == 0
    y = yd.cpu().numpy()
    assert y[-2] == np.inf and y[-1] == 0.0
    err = np.abs(y[:-2].astype(np.float64) * np.sqrt(x[:-2].astype(np.float64)) - 1) * 2.0 ** 24
    assert err.max() <= 1.5, float(err.max())


def tiny_hinge():
    b = I._Builder("tiny")
    b.link(-1, I.REVOLUTE, axis=(0, 1, 0), mass=0.0, com=(0, 0, 0), inertia=1e-40 * np.eye(3))
    return b.finish(act_dof=[0], act_gear=[1.0], dt=I.CONTROL_DT, substeps=2)


def short_muscle():
    """45 muscles, one between two points of a link 1e-20 m apart."""
    rng = np.random.default_rng(1)
    b = I._Builder("short")
    m, c, J = I.capsule_mass_inertia(0.04, (0, 0, 0), (0, 0, -0.3), 1000.0)
    links = [b.link(-1, I.REVOLUTE, axis=(0, 1, 0), mass=m, com=c, inertia=J)]
    for _ in range(3):
        links.append(b.link(links[-1], I.REVOLUTE, axis=(1, 0, 0), pos=(0, 0, -0.3), mass=m, com=c, inertia=J))
    b.muscle(50.0, [(links[0], np.array([1e-20, 0, 0])), (links[0], np.zeros(3))])
    for k in range(44):
        b.muscle(30.0, [(lk, rng.uniform(-0.05, 0.05, 3) + np.array([0, 0, -0.15])) for lk in links[k % 3:k % 3 + 2]])
    return b.finish(act_dof=[], act_gear=[], dt=I.CONTROL_DT, substeps=4, armature=0.05, damping=0.5)


@pytest.mark.parametrize("spec", [False, True])
@pytest.mark.parametrize("make", [tiny_hinge, short_muscle, sliding_ball])
def test_steps_at_the_ends_of_the_range(make, spec):
    from paper_2204_07137_gb300.sim import Simulator
    m, N = make(), 5
    q, qd = I.random_state(m, N, 2, pos_scale=0.1, vel_scale=0.1)
    a = np.full((m.na, N), 0.5 if m.n_muscles else 0.0, np.float32)
    if make is sliding_ball:
        q, qd = np.zeros((7, N)), np.zeros((6, N))
        q[2], q[6], qd[3] = 0.099, 1.0, 1e20
    out = []
    for lane_form in (True, False):
        sim = Simulator([(m, N)] + ([] if lane_form else [(many_links(), 1)]), form="batched", h_max=1)
        if spec and lane_form:
            sim.specialize()
        x = [torch.cat([T(v)] + ([] if lane_form else [torch.zeros(1, device="cuda")])) for v in (q, qd, a)]
        y = sim.step(*x)
        torch.cuda.synchronize()
        assert sim.status() == 0      # no non-finite state
        out.append([v[:k * N].cpu().numpy() for v, k in zip(y, (m.nq, m.nv))])
    for u, v in zip(*out):
        np.testing.assert_allclose(u, v, rtol=1e-5, atol=1e-6)
