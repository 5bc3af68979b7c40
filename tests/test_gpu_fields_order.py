"""wdlb_fields returns the very forces that the time step uses: its C equals,
bit for bit, the C that one step from the same state keeps for the next (the
saved state's C_prev).  Generic shell kernel with a node's pairs split over four
warps (any closure, storage and collision arithmetic) and unsplit, and the tiled
kernel; walls and periodic boxes, node counts off the kernels' block sizes.
The saved state ends with C_prev (three arrays), t_prev and the storage scale,
each padded to 64 nodes."""
import numpy as np
import pytest

from paper_1304_7880_gb300 import synth

pytestmark = pytest.mark.gpu

# lattice, sigma, walls, storage, shell rule, closure, collision
CASES = [
    ((7, 9, 33), 8.0, True, "f32", "full", "CS", "fp32"),
    ((9, 8, 31), 4.0, True, "f32", "full", "PY", "fp32"),
    ((6, 5, 21), 4.0, True, "f32", "full", "CS", "dw"),
    ((5, 7, 29), 5.0, True, "f64", "full", "ONE", "fp32"),
    ((11, 6, 13), 8.0, False, "f16", "full", "CS", "fp32"),
    ((6, 5, 21), 4.0, True, "f32", "compact", "CS", "fp32"),
    ((9, 8, 23), 4.0, True, "f64", "compact", "CS", "fp32"),
    ((17, 15, 9), 1.5, False, "f32", "full", "CS", "fp32"),
    ((10, 9, 27), 4.0, True, "f32", "full", "CS", "fp32"),       # tiled
    ((12, 9, 35), 6.0, False, "f16", "full", "CS", "fp32"),      # tiled
]


@pytest.fixture(scope="module")
def w():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1304_7880_gb300 import build, wdlb
    build.build()
    return wdlb


@pytest.mark.parametrize("lat,sigma,walls,storage,rule,closure,collision", CASES)
def test_fields_forces_are_the_steps(w, lat, sigma, walls, storage, rule, closure, collision):
    n, u = synth.uniform_with_noise(*lat, 0.4 / sigma ** 3, 2e-2, 5, walls)
    ctx = w.wdlb_create(lat, sigma, walls, 1.0, (1e-5, 0.0, 0.0), storage=storage, shell_rule=rule, closure=closure,
                        collision=collision)
    w.wdlb_init_fields(ctx, n, u)
    w.wdlb_step(ctx, 3)
    C = w.wdlb_fields(ctx)[1]
    w.wdlb_step(ctx, 1)
    T = np.float64 if storage == "f64" else np.float32
    pad = (n.size + 63) // 64 * 64
    prev = w.wdlb_save_state(ctx)[-5 * pad * T().itemsize:].view(T)[:3 * pad].reshape(3, pad)[:, :n.size]
    prev = prev.reshape((3,) + n.shape).astype(np.float64)
    m = slice(1, -1) if walls else slice(None)
    assert np.abs(C[:, m]).max() > 0.0
    assert np.array_equal(C[:, m], prev[:, m])
    w.wdlb_destroy(ctx)
