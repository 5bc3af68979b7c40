"""Rounding of the pair weights on the device (tests/pair_arith/pair_arith.cu
inlines the step kernels' own functions) against FP64 of the same inputs.

FP32: the weights Q+, Q- and the difference 2 (Q+ - Q-) are held to the
closures written in s = 1 - chi_mid with every operation correctly rounded
(numpy, multiply-adds fused), over bulk-like and wall-like pairs.  Bound on the
rms relative error: 1.15 times that reference's.  With the hardware's reciprocal
in it, whose error may spread over two ulps, the form in s comes to 1.11 to
1.145 times (numpy, reciprocals off by up to 0.9 ulp).  Forming a = 1/s first
and then a^2 and a^3 carries the reciprocal's error 2.6 times into the weight:
1.25 to 1.29 (Carnahan-Starling) with rounded reciprocals already, 2.0 with such
ones.

FP64: the worst relative error of a weight is ten half-ulps (three from s, two
from s^3, two from its reciprocal, one each from the closure's multiply-add, the
density and the product).  fast_rcp<double> refines an approximation good to
2^-19 by the geometric series of 1/(1 - e) cut after e^2: what it drops is
e^3 < 2^-57, so its error stays below 0.57 ulp."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.join(os.path.dirname(os.path.abspath(__file__)), "pair_arith")


@pytest.fixture(scope="module")
def lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1304_7880_gb300 import build
    out = os.path.join(HERE, "_build", "pair_arith.so")
    os.makedirs(os.path.dirname(out), exist_ok=True)
    tmp = out + ".tmp%d" % os.getpid()
    subprocess.check_call([build.nvcc(), *build.ARCH, *build.FLAGS, "-shared", "-o", tmp,
                           os.path.join(HERE, "pair_arith.cu"), "-lcudart"])
    os.replace(tmp, out)
    return ctypes.CDLL(out)


def _states(kind, count, dtype):
    """s0, noff, dh+, dn+, dh-, dn- of pairs as a lattice has them: smooth
    deviations (bulk), or densities from zero to 2.3 n_off beside a wall."""
    r = np.random.RandomState(11 if kind == "bulk" else 12)
    chi = r.uniform(0.05, 0.33, count)                       # packing fraction, n* up to 0.6
    noff, hoff = chi / 33.5, 0.5 * chi
    dh0 = (0.02 if kind == "bulk" else 0.3) * hoff * r.uniform(-1, 1, count)
    cols = [1.0 - (hoff + dh0) - hoff, noff]
    for _ in range(2):
        cols.append(hoff * (1e-2 * r.randn(count) if kind == "bulk" else r.uniform(-1.0, 0.4, count)))
        cols.append(noff * (1e-2 * r.randn(count) if kind == "bulk" else r.uniform(-1.0, 1.3, count)))
    return np.ascontiguousarray(np.stack(cols, 1).astype(dtype))


def _run(fn, closure, x):
    out = np.empty((len(x), 3), dtype=x.dtype)
    assert fn(closure, len(x), x.ctypes.data_as(ctypes.c_void_p), out.ctypes.data_as(ctypes.c_void_p)) == 0
    return out


def _weights(closure, cols, one, fma):
    """Q+, Q-, 2 (Q+ - Q-) in the closures' form in s; one: the number 1 of the arithmetic."""
    s0, noff, hp, dp, hm, dm = cols
    np_, nm, sp, sm = noff + dp, noff + dm, s0 - hp, s0 - hm
    spm, sp2, sm2 = sp * sm, sp * sp, sm * sm
    if closure == 0:
        rp, rm = one / (sp2 * sp), one / (sm2 * sm)
        gp, gm = fma(sp, rp, rp), fma(sm, rm, rm)
        gd = (hp - hm) * ((sp2 + sm2) + fma(spm, sp + sm, spm)) * (rp * rm)
    else:
        rp, rm = one / sp2, one / sm2
        three = one + one + one
        gp, gm = fma(-sp, rp, three * rp), fma(-sm, rm, three * rm)
        gd = (hp - hm) * fma(three, sp + sm, -spm) * (rp * rm)
    return gp * np_, gm * nm, fma(gp + gm, dp - dm, gd * (np_ + nm)), (gp + gm, gd, np_ + nm, dp - dm)


def _fma32(a, b, c):
    return (a.astype(np.float64) * b + c.astype(np.float64)).astype(np.float32)


@pytest.mark.parametrize("kind", ["bulk", "wall"])
@pytest.mark.parametrize("closure", [0, 1])
def test_fp32_weights_round_no_worse_than_the_form_in_s(lib, closure, kind):
    x = _states(kind, 1 << 20, np.float32)
    got = _run(lib.pair_weights_f32, closure, x)
    ref = _weights(closure, list(x.T), np.float32(1), _fma32)
    exact = _weights(closure, list(x.T.astype(np.float64)), 1.0, lambda a, b, c: a * b + c)
    gs, gd, ns, dn = exact[3]
    # Q relative to itself, the difference relative to the size of its two parts
    for k, scale in ((0, np.abs(exact[0])), (1, np.abs(exact[1])), (2, np.abs(gs * dn) + np.abs(gd * ns))):
        ok = scale > 1e-6 * scale.max()
        e_got = np.sqrt(np.mean(((got[:, k] - exact[k])[ok] / scale[ok]) ** 2))
        e_ref = np.sqrt(np.mean(((ref[k] - exact[k])[ok] / scale[ok]) ** 2))
        print("closure %d %s output %d: rms error %.3e, form in s %.3e, ratio %.3f" % (closure, kind, k, e_got, e_ref, e_got / e_ref))
        assert e_got <= 1.15 * e_ref


@pytest.mark.parametrize("kind", ["bulk", "wall"])
@pytest.mark.parametrize("closure", [0, 1])
def test_fp64_weights_are_within_ten_half_ulps(lib, closure, kind):
    x = _states(kind, 2000, np.float64)
    got = _run(lib.pair_weights_f64, closure, x)
    for i in range(len(x)):
        e = _weights(closure, [Fraction(v) for v in x[i].tolist()], Fraction(1), lambda a, b, c: a * b + c)
        for k in (0, 1):
            assert abs(Fraction(float(got[i, k])) - e[k]) <= 10 * Fraction(1, 2 ** 53) * abs(e[k])


def test_fp64_reciprocal_error(lib):
    r = np.random.RandomState(3)
    x = np.concatenate([r.uniform(0.02, 1.0, 4000), r.uniform(0.02, 1.0, 2000) ** 3, 2.0 ** r.uniform(-20, 2, 2000),
                        1.0 + np.arange(64) * 2.0 ** -52, 1.0 - np.arange(64) * 2.0 ** -53])
    out = np.empty_like(x)
    assert lib.rcp_f64(len(x), x.ctypes.data_as(ctypes.c_void_p), out.ctypes.data_as(ctypes.c_void_p)) == 0
    worst = 0.0
    for a, b in zip(x.tolist(), out.tolist()):
        worst = max(worst, float(abs(Fraction(b) - 1 / Fraction(a)) / Fraction(float(np.spacing(1.0 / a)))))
    print("fast_rcp<double>: %.4f ulp" % worst)
    assert worst <= 0.57
