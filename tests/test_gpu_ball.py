"""The smeared density (FP64, through wdlb_fields) on bricks whose columns are
shared between outputs, against the oracle at 1e-12: sigma 3, 4, 6, 8 (compiled
balls; sigma 8 in FP64 keeps the unpadded brick), lattices ragged against the 8^3
brick, axes shorter than the ball and walls."""
import numpy as np
import pytest

from paper_1304_7880_gb300 import synth

pytestmark = pytest.mark.gpu

CASES = [((9, 8, 7), 8.0, False), ((17, 9, 21), 6.0, True), ((1, 3, 12), 8.0, True), ((2, 1, 3), 6.0, False),
         ((8, 8, 9), 3.0, True), ((11, 18, 5), 4.0, False), ((8, 16, 10), 8.0, True)]


@pytest.fixture(scope="module")
def w():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1304_7880_gb300 import build, wdlb
    build.build()
    return wdlb


@pytest.mark.parametrize("lat,sigma,walls", CASES)
def test_smeared_density_matches_the_oracle(w, oracle_mod, lat, sigma, walls):
    n, u = synth.uniform_with_noise(*lat, 0.3 / sigma ** 3, 0.2, 8, walls)
    ctx = w.wdlb_create(lat, sigma, walls, 1.0, storage="f64")
    w.wdlb_init_fields(ctx, n, u)
    o = oracle_mod.Oracle(*lat, walls, sigma, 1.0, (0.0, 0.0, 0.0))
    o.init(n, u)
    m = slice(1, -1) if walls else slice(None)
    np.testing.assert_allclose(w.wdlb_fields(ctx)[0][m], o.fields()[0][m], rtol=1e-12)
