"""Every form of the shell kernels, each checked to be the one that runs
(wdlb_shell_info, wdlb_batch_shell_info).

The tiled full-shell kernel's form for launches of at most one block per SM
gives the bits of the other form, for every sigma and tile shape, FP32 and FP16
storage and the double-word collision.  The generic kernel with a node's pairs
split over four warps and unsplit, in FP32, FP16 and with the double-word
collision, closures PY and ONE among them, agrees with the FP64 oracle after
four steps within the library's bounds for noisy states: FP32 1e-5 of n and of
max|u|, FP16 1e-6 and 5e-3."""
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


@pytest.mark.parametrize("storage,collision,walls", [("f32", "fp32", True), ("f32", "fp32", False),
                                                     ("f16", "fp32", False), ("f32", "dw", True)])
@pytest.mark.parametrize("tile", [0, 1, 2])
@pytest.mark.parametrize("sigma", [3.0, 4.0, 6.0])
def test_roomy_form_on_every_tile_shape(w, sigma, tile, storage, collision, walls):
    lat, g, kw = (17, 12, 21), (1e-5, 0.0, 0.0), dict(storage=storage, collision=collision, tile=tile)
    n, u = synth.uniform_with_noise(*lat, 0.4 / sigma ** 3, 2e-2, 3, walls)
    ctx = w.wdlb_create(lat, sigma, walls, 1.0, g, **kw)
    w.wdlb_init_fields(ctx, n, u)
    w.wdlb_step(ctx, 3)
    assert w.wdlb_tile_info(ctx) == (True, tile) and w.wdlb_shell_info(ctx) == (False, True)
    b = w.wdlb_batch_create(2, 512 << 20, **kw)
    slot = w.wdlb_batch_add(b, lat, sigma, walls, 1.0, g, n, u)
    w.wdlb_batch_add(b, (64, 64, 64), sigma, walls, 1.0, g,
                     *synth.uniform_with_noise(64, 64, 64, 0.4 / sigma ** 3, 1e-3, 4, walls))
    w.wdlb_batch_step(b, 3)
    assert w.wdlb_batch_shell_info(b) == (1, 0, 0)
    assert np.array_equal(w.wdlb_get_populations(ctx), w.wdlb_get_populations(w.wdlb_batch_context(b, slot)))
    w.wdlb_batch_destroy(b)
    w.wdlb_destroy(ctx)


# lattice, sigma, walls, storage, shell rule, closure, collision, split
GENERIC = [
    ((7, 9, 33), 8.0, True, "f32", "full", "CS", "fp32", True),
    ((3, 1, 31), 8.0, False, "f32", "full", "CS", "fp32", True),
    ((9, 8, 31), 4.0, False, "f32", "full", "PY", "fp32", True),
    ((5, 7, 29), 5.0, True, "f32", "full", "ONE", "fp32", True),
    ((6, 5, 21), 4.0, True, "f32", "full", "CS", "dw", True),
    ((11, 6, 23), 8.0, False, "f16", "full", "CS", "fp32", True),
    ((9, 8, 23), 4.0, False, "f16", "full", "PY", "fp32", True),
    ((16, 9, 25), 8.0, False, "f32", "compact", "CS", "fp32", False),
    ((9, 8, 23), 4.0, True, "f32", "compact", "PY", "dw", False),
    ((17, 15, 9), 1.5, False, "f32", "full", "CS", "fp32", False),
    ((9, 8, 23), 3.0, True, "f64", "compact", "CS", "fp32", False),
    ((9, 8, 23), 4.0, True, "f64", "full", "ONE", "fp32", True),
]
TOL = {"f64": (1e-10, 1e-10), "f32": (1e-5, 1e-5), "f16": (1e-6, 5e-3)}


@pytest.mark.parametrize("lat,sigma,walls,storage,rule,closure,collision,split", GENERIC)
def test_generic_forms_match_the_oracle(w, oracle_mod, lat, sigma, walls, storage, rule, closure, collision, split):
    n, u = synth.uniform_with_noise(*lat, 0.3 / sigma ** 3, 2e-2, 5, walls)
    u = 1e-3 * np.random.RandomState(5).standard_normal(u.shape)
    if walls:
        u[:, 0] = u[:, -1] = 0.0
    g = (1e-5, 0.0, 0.0)
    ctx = w.wdlb_create(lat, sigma, walls, 1.0, g, storage=storage, shell_rule=rule, closure=closure,
                        collision=collision)
    w.wdlb_init_fields(ctx, n, u)
    assert w.wdlb_tile_info(ctx)[0] is False and w.wdlb_shell_info(ctx) == (split, False)
    o = oracle_mod.Oracle(*lat, walls, sigma, 1.0, g, closure=closure, shell_rule=rule)
    o.init(n, u)
    w.wdlb_step(ctx, 4)
    o.step(4)
    n_g, u_g = w.wdlb_moments(ctx)
    n_o, u_o = o.moments()
    m = slice(1, -1) if walls else slice(None)
    tn, tu = TOL[storage]
    np.testing.assert_allclose(n_g[m], n_o[m], rtol=tn)
    np.testing.assert_allclose(u_g[:, m], u_o[:, m], rtol=0, atol=tu * np.abs(u_o[:, m]).max())
    w.wdlb_destroy(ctx)


@pytest.mark.parametrize("storage,closure", [("f64", "CS"), ("f32", "PY")])
def test_without_interactions_nothing_is_split(w, oracle_mod, storage, closure):
    lat = (9, 8, 23)
    n, u = synth.uniform_with_noise(*lat, 0.3 / 64, 2e-2, 7, True)
    ctx = w.wdlb_create(lat, 4.0, True, 1.0, (1e-5, 0.0, 0.0), storage=storage, closure=closure, interactions=False)
    w.wdlb_init_fields(ctx, n, u)
    assert w.wdlb_shell_info(ctx) == (False, False)
    o = oracle_mod.Oracle(*lat, True, 4.0, 1.0, (1e-5, 0.0, 0.0), closure=closure, interactions=False)
    o.init(n, u)
    w.wdlb_step(ctx, 4)
    o.step(4)
    (n_g, u_g), (n_o, u_o) = w.wdlb_moments(ctx), o.moments()
    tn, tu = TOL[storage]
    np.testing.assert_allclose(n_g[1:-1], n_o[1:-1], rtol=tn)
    np.testing.assert_allclose(u_g[:, 1:-1], u_o[:, 1:-1], rtol=0, atol=tu * np.abs(u_o[:, 1:-1]).max())
    w.wdlb_destroy(ctx)


def test_batch_of_split_and_unsplit_groups(w):
    b = w.wdlb_batch_create(3, 64 << 20, storage="f32")
    for lat, sigma in (((9, 8, 25), 8.0), ((8, 8, 17), 1.5), ((9, 11, 25), 4.0)):
        w.wdlb_batch_add(b, lat, sigma, True, 1.0, (1e-5, 0.0, 0.0),
                         *synth.uniform_with_noise(*lat, 0.3 / sigma ** 3, 1e-2, 6, True))
    w.wdlb_batch_step(b, 2)
    assert w.wdlb_batch_shell_info(b) == (3, 1, 1)      # one split, one unsplit, one tiled (roomy)
    w.wdlb_batch_destroy(b)
