"""One batch of pores that run different kernels in every phase (compiled and
run-time balls; the shell kernel tiled, generic with split pairs and generic
unsplit) gives each pore the bits it has alone, through a removal; FP32, FP64
and the double-word collision."""
import numpy as np
import pytest

from paper_1304_7880_gb300 import synth

pytestmark = pytest.mark.gpu

# lattice, sigma
PORES = [((9, 11, 25), 4.0), ((6, 5, 21), 4.0), ((13, 9, 19), 3.5), ((8, 8, 17), 1.5), ((10, 7, 33), 8.0),
         ((12, 9, 23), 3.0), ((7, 9, 27), 5.0)]


@pytest.fixture(scope="module")
def w():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1304_7880_gb300 import build, wdlb
    build.build()
    return wdlb


@pytest.mark.parametrize("storage,collision", [("f32", "fp32"), ("f64", "fp32"), ("f32", "dw")])
def test_mixed_kernels_in_one_batch_equal_alone(w, storage, collision):
    g = (1e-5, 0.0, 0.0)
    b = w.wdlb_batch_create(len(PORES), 128 << 20, storage=storage, collision=collision)
    init = [synth.uniform_with_noise(*lat, 0.3 / sigma ** 3, 2e-2, 30 + k, True) for k, (lat, sigma) in enumerate(PORES)]
    slots = [w.wdlb_batch_add(b, lat, sigma, True, 1.0, g, n, u) for (lat, sigma), (n, u) in zip(PORES, init)]
    w.wdlb_batch_step(b, 3)
    w.wdlb_batch_remove(b, slots[0])
    w.wdlb_batch_step(b, 3)
    for (lat, sigma), (n, u), slot in list(zip(PORES, init, slots))[1:]:
        ctx = w.wdlb_create(lat, sigma, True, 1.0, g, storage=storage, collision=collision)
        w.wdlb_init_fields(ctx, n, u)
        w.wdlb_step(ctx, 6)
        assert np.array_equal(w.wdlb_get_populations(ctx), w.wdlb_get_populations(w.wdlb_batch_context(b, slot))), sigma
        w.wdlb_destroy(ctx)
    w.wdlb_batch_destroy(b)
