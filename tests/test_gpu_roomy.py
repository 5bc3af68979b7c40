"""The tiled full-shell kernel has a second form for launches of at most one
block per SM (more registers, four couples per iteration).  A pore alone runs
it; the same pore in a batch with a 64^3 box (more blocks than SMs) runs the
other one.  Both sum the same terms in the same order: bit-identical
populations, for every sigma and tile shape, with and without walls, also with
the double-word collision."""
import numpy as np
import pytest

from paper_1304_7880_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def w():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1304_7880_gb300 import build, wdlb
    build.build()
    return wdlb


@pytest.mark.parametrize("collision", ["fp32", "dw"])
@pytest.mark.parametrize("sigma", [3.0, 4.0, 6.0])
@pytest.mark.parametrize("walls", [True, False])
def test_roomy_form_gives_the_same_bits(w, sigma, walls, collision):
    if collision == "dw" and not walls:
        pytest.skip("the double-word collision is for slits")
    lat, g = (17, 12, 29), (1e-5, 0.0, 0.0)
    n, u = synth.uniform_with_noise(*lat, 0.4 / sigma ** 3, 2e-2, 3, walls)
    ctx = w.wdlb_create(lat, sigma, walls, 1.0, g, storage="f32", collision=collision)
    w.wdlb_init_fields(ctx, n, u)
    w.wdlb_step(ctx, 5)
    b = w.wdlb_batch_create(2, 512 << 20, storage="f32", collision=collision)
    slot = w.wdlb_batch_add(b, lat, sigma, walls, 1.0, g, n, u)
    bn, bu = synth.uniform_with_noise(64, 64, 64, 0.4 / sigma ** 3, 1e-3, 4, walls)
    w.wdlb_batch_add(b, (64, 64, 64), sigma, walls, 1.0, g, bn, bu)
    w.wdlb_batch_step(b, 5)
    assert np.array_equal(w.wdlb_get_populations(ctx), w.wdlb_get_populations(w.wdlb_batch_context(b, slot)))
    w.wdlb_batch_destroy(b)
