"""Slits with the double-word collision, the accuracy option, give the same bits
from one version of the library to the next: their pairs are summed in table
order with the weights in s.  (Summed as mirror couples, the converged 161-node
slit at n* 0.3 was 9.3e-6 off on u_x instead of 4.8e-6, against a bound of 1e-5.)
tests/golden/dw_bits.txt holds, per case, the SHA-256 of the populations and of n
and u after six steps, recorded on a GB300 (sm_103a, nvcc 13.0): the tiled kernel
at sigma 3, 4 and 6 on every tile shape, full and compact shell, ragged slits."""
import hashlib
import os

import numpy as np
import pytest

from paper_1304_7880_gb300 import synth

pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "dw_bits.txt")
CASES = {"s%d_%s" % (sigma, rule): (lat, float(sigma), rule)
         for sigma, lat in ((3, (13, 11, 22)), (4, (10, 9, 27)), (6, (12, 9, 35))) for rule in ("full", "compact")}


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
    n, _ = synth.uniform_with_noise(*lat, 0.4375 / sigma ** 3, 0.015625, 21, True)
    u = 0.0009765625 * (2.0 * synth.uniform01(22, 3 * n.size).reshape((3,) + n.shape) - 1.0)
    u[:, 0] = u[:, -1] = 0.0
    ctx = w.wdlb_create(lat, sigma, True, 1.0, (2.0 ** -17, 0.0, 0.0), storage="f32", collision="dw",
                        shell_rule=rule, tile=tile, autotune=False)
    w.wdlb_init_fields(ctx, n, u)
    w.wdlb_step(ctx, 6)
    h = hashlib.sha256(np.ascontiguousarray(w.wdlb_get_populations(ctx)[:, 1:-1]).tobytes())
    n_g, u_g = w.wdlb_moments(ctx)
    for a in (n_g[1:-1], u_g[:, 1:-1]):
        h.update(np.ascontiguousarray(a).tobytes())
    w.wdlb_destroy(ctx)
    return h.hexdigest()


@pytest.mark.parametrize("tile", [0, 1, 2])
@pytest.mark.parametrize("name", sorted(CASES))
def test_dw_slit_keeps_its_bits(w, name, tile):
    want = dict(line.split() for line in open(GOLDEN))
    assert digest(w, *CASES[name], tile) == want[name]
