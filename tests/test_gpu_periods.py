"""A periodic state has the same bits on a box of one period and on a box of
five: the kernel that serves a node in FP32 does not depend on the size of its
lattice.  Generic shell kernel (sigma 8, Percus-Yevick, sigma 1.5: compact and
full shells), node counts on both sides of 24 576, where small compact lattices
once took the kernel that splits a node's pairs, which is slower once a batch of
them fills the GPU."""
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


@pytest.mark.parametrize("sigma,rule,closure", [(8.0, "compact", "CS"), (4.0, "compact", "PY"), (1.5, "full", "CS"),
                                                (8.0, "full", "CS")])
def test_one_period_and_five_agree(w, sigma, rule, closure):
    n, u = synth.uniform_with_noise(16, 16, 20, 0.4 / sigma ** 3, 2e-2, 5, False)
    pops = []
    for k in (1, 5):
        ctx = w.wdlb_create((16, 16, 20 * k), sigma, False, 1.0, (1e-5, 0.0, 0.0), shell_rule=rule, closure=closure,
                            n_ref=0.4 / sigma ** 3)
        w.wdlb_init_fields(ctx, np.tile(n, (k, 1, 1)), np.tile(u, (1, k, 1, 1)))
        w.wdlb_step(ctx, 4)
        pops.append(w.wdlb_get_populations(ctx))
        w.wdlb_destroy(ctx)
    assert np.array_equal(np.tile(pops[0], (1, 5, 1, 1)), pops[1])
