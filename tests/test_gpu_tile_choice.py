"""The tile shape that a pore gets by default depends on its kernel and not on
the probe's noise: full-shell sigma-4 pores of any nz share one shape, so a batch
of them keeps one shell launch per step, and a persistent batch of them is served
by the persistent kernel (one launch per call) with the autotuner on as with it
off.  Compact-shell pores, which a probe puts on another shape, are served by it
unprobed."""
import pytest

from paper_1304_7880_gb300 import synth

pytestmark = pytest.mark.gpu

NZ = (13, 24, 33, 41, 64, 80, 81, 121, 128, 161)


@pytest.fixture(scope="module")
def w():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1304_7880_gb300 import build, wdlb
    build.build()
    return wdlb


def _launches(w, nz, walls, steps, **kw):
    w.wdlb_autotune_reset()
    b = w.wdlb_batch_create(len(nz), 256 << 20, storage="f32", **kw)
    for k in nz:
        n, u = synth.uniform_with_noise(16, 12, k, 0.3 / 64, 1e-3, k, walls)
        w.wdlb_batch_add(b, (16, 12, k), 4.0, walls, 1.0, (1e-6, 0.0, 0.0), n, u)
    w.wdlb_batch_step(b, 2)
    at = w.wdlb_batch_launch_count(b)
    w.wdlb_batch_step(b, steps)
    got = w.wdlb_batch_launch_count(b) - at
    w.wdlb_batch_destroy(b)
    return got


@pytest.mark.parametrize("walls", [True, False])
def test_full_shell_pores_share_one_shell_launch(w, walls):
    assert _launches(w, NZ, walls, 4) == 4 * 3


@pytest.mark.parametrize("rule,autotune", [("full", True), ("full", False), ("compact", False)])
def test_persistent_batch_runs_the_persistent_kernel(w, rule, autotune):
    assert _launches(w, (13, 41, 80), True, 6, persistent=True, shell_rule=rule, autotune=autotune) == 1
