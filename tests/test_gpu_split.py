"""The generic shell kernel with a node's pairs split over four warps (full
shells, and any shell on small lattices) and unsplit (compact shells on larger
ones), in FP64 against the oracle at 1e-10: node counts around the 32 nodes of a
block and the 256 of a work item, axes shorter than the shell (indices that wrap
more than once), walls, and both sides of the node count where the compact
shell stops splitting."""
import numpy as np
import pytest

from paper_1304_7880_gb300 import synth

pytestmark = pytest.mark.gpu

CASES = [
    ((1, 1, 31), 4.0, False, "full"),
    ((3, 1, 11), 8.0, False, "full"),
    ((5, 3, 17), 4.0, True, "full"),       # 255 nodes
    ((4, 4, 16), 3.0, True, "compact"),    # 256
    ((1, 257, 1), 2.0, False, "full"),
    ((7, 9, 33), 6.0, True, "full"),
    ((32, 32, 24), 4.0, False, "compact"),  # 24 576: split
    ((31, 29, 28), 4.0, True, "compact"),   # 25 172: unsplit
]


@pytest.fixture(scope="module")
def w():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1304_7880_gb300 import build, wdlb
    build.build()
    return wdlb


@pytest.mark.parametrize("lat,sigma,walls,rule", CASES)
def test_split_sums_match_the_oracle(w, oracle_mod, lat, sigma, walls, rule):
    nx, ny, nz = lat
    n, u = synth.uniform_with_noise(nx, ny, nz, 0.3 / sigma ** 3, 2e-2, 5, walls)
    u = 1e-3 * np.random.default_rng(5).standard_normal(u.shape)
    if walls:
        u[:, 0] = u[:, -1] = 0.0
    g = (1e-5, 0.0, 0.0)
    ctx = w.wdlb_create(lat, sigma, walls, 1.0, g, storage="f64", shell_rule=rule)
    w.wdlb_init_fields(ctx, n, u)
    o = oracle_mod.Oracle(nx, ny, nz, walls, sigma, 1.0, g, shell_rule=rule)
    o.init(n, u)
    w.wdlb_step(ctx, 4)
    o.step(4)
    n_g, u_g = w.wdlb_moments(ctx)
    n_o, u_o = o.moments()
    m = slice(1, -1) if walls else slice(None)
    np.testing.assert_allclose(n_g[m], n_o[m], rtol=1e-10)
    np.testing.assert_allclose(u_g[:, m], u_o[:, m], rtol=0, atol=1e-10 * np.abs(u_o[:, m]).max())
