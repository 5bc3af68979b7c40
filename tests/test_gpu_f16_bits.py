"""FP16-storage boxes give the same bits from one version of the library to the
next: their stored populations turn a last bit of the FP32 arithmetic into 1e-4
of u, so any reordering shows in every result.  tests/golden/f16_bits.txt holds,
per case, the SHA-256 of the populations and of n and u after six steps,
recorded on a GB300 (sm_103a, nvcc 13.0) with pairs in table order, closures in
s and the collision direction by direction: the tiled kernel at sigma 3, 4 and 6
on every tile shape, full and compact shell, ragged boxes."""
import hashlib
import os

import numpy as np
import pytest

from paper_1304_7880_gb300 import synth

pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "f16_bits.txt")
CASES = {"s%d_%s" % (sigma, rule): (lat, float(sigma), rule)
         for sigma, lat in ((3, (13, 11, 19)), (4, (17, 9, 26)), (6, (14, 19, 24))) for rule in ("full", "compact")}


@pytest.fixture(scope="module")
def w():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1304_7880_gb300 import build, wdlb
    build.build()
    return wdlb


def digest(w, lat, sigma, rule, tile):
    # products of exact binary draws only: the same inputs on every machine
    n, _ = synth.uniform_with_noise(*lat, 0.4375 / sigma ** 3, 0.015625, 21, False)
    u = 0.015625 * (2.0 * synth.uniform01(22, 3 * n.size).reshape((3,) + n.shape) - 1.0)
    ctx = w.wdlb_create(lat, sigma, False, 1.0, storage="f16", shell_rule=rule, tile=tile, autotune=False)
    w.wdlb_init_fields(ctx, n, u)
    w.wdlb_step(ctx, 6)
    h = hashlib.sha256(w.wdlb_get_populations(ctx).tobytes())
    for a in w.wdlb_moments(ctx):
        h.update(np.ascontiguousarray(a).tobytes())
    w.wdlb_destroy(ctx)
    return h.hexdigest()


@pytest.mark.parametrize("tile", [0, 1, 2])
@pytest.mark.parametrize("name", sorted(CASES))
def test_f16_box_keeps_its_bits(w, name, tile):
    want = dict(line.split() for line in open(GOLDEN))
    assert digest(w, *CASES[name], tile) == want[name]
