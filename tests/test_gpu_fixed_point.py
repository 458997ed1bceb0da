"""The fixed-point exponentials and logarithm of the rates and properties against longer arithmetic.

Bounds, in units in the last place of the result (the last rounding is half a unit):
* 2^(x/256): the argument is cut at 2^-45, exact from |x| = 256 on (FP64 spacing), below that a relative
  error of 2^-45 ln2/256 = 0.35 2^-52, up to 0.7 units for a mantissa near 2; table, polynomial and products
  (63 fraction bits) below 0.05 units: 0.55 units from 256 on, 1.25 below;
* exp(x): the product x log2(e) is cut at 2^-53 of a factor of 2^(1/256) likewise; x itself at 2^-53, exact
  from |x| = 1 on: 1.25 units from 1 on, and below 1 another 0.35 log2(e) of a unit: 2.25;
* log(x): the rounding of the mantissa's part and of the two multiply-adds: 1.5 units; near 1 CUDA's log,
  1 unit.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LD = np.longdouble


def _run(mechs, which, x):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2402_18858_gb300 import build, chem as lc
    build.build()
    gm = lc.chem_load_mech(mechs["h2_9"][1])
    xd = torch.as_tensor(np.ascontiguousarray(x), device="cuda")
    y = torch.empty_like(xd)
    lc.chem_selftest_fix(gm, which, xd, y)
    return y.cpu().numpy()


def _ulp(y, ref):
    return np.abs((y.astype(LD) - ref) / np.spacing(ref.astype(np.float64)).astype(LD)).astype(np.float64)


def _near(rng, n, lo, hi):   # both signs, magnitudes spread over their logarithm
    return rng.choice([-1.0, 1.0], n) * 10.0 ** rng.uniform(np.log10(lo), np.log10(hi), n)


@pytest.mark.parametrize("which", [1, 2])
def test_exp256(mechs, which):
    rng = np.random.default_rng(1)
    x = np.concatenate([rng.uniform(-261484.9, 261484.9, 40000), _near(rng, 40000, 256.0, 261484.0),
                        256.0 * rng.integers(-1000, 1000, 2000), rng.integers(-260000, 260000, 20000).astype(float)])
    small = np.concatenate([_near(rng, 40000, 1e-320, 255.9), [0.0, -0.0, 1.0, -1.0, 0.5, 255.0, 2.0 ** -45, -2.0 ** -46]])
    sign = LD(1 if which == 1 else -1)
    big = np.abs(x) >= 256.0
    x = x[big]
    for a, bound in ((x, 0.55), (small, 1.25)):
        y = _run(mechs, which, a)
        u = _ulp(y, np.exp2(sign * a.astype(LD) / LD(256)))
        print("2^(x/256)", which, "worst", u.max(), "at", a[np.argmax(u)])
        assert u.max() <= bound, (u.max(), a[np.argmax(u)])
    assert (_run(mechs, which, np.array([0.0, -0.0])) == 1.0).all()


def test_exp256_ends(mechs):
    x = np.array([np.nan, np.inf, -np.inf, -261486.0, -3e5, 262144.0, 1e300, -1e300])
    y = _run(mechs, 1, x)
    assert np.isnan(y[0]) and y[1] == np.inf and y[5] == np.inf and y[6] == np.inf
    assert (y[[2, 3, 4, 7]] == 0.0).all()
    x = np.array([261485.0, 262143.9, -261485.0, -261485.59])     # the last finite results
    u = _ulp(_run(mechs, 1, x), np.exp2(x.astype(LD) / LD(256)))
    assert u.max() <= 0.55


def test_exp(mechs):
    rng = np.random.default_rng(2)
    for a, bound in ((np.concatenate([rng.uniform(-707.9, 709.7, 60000), _near(rng, 60000, 1.0, 700.0)]), 1.25),
                     (np.concatenate([_near(rng, 60000, 1e-320, 0.999), [0.0, -0.0, 2.0 ** -53, -2.0 ** -54]]), 2.25)):
        a = a[(np.abs(a) >= 1.0) == (bound < 2.0)]
        u = _ulp(_run(mechs, 0, a), np.exp(a.astype(LD)))
        print("exp worst", u.max(), "at", a[np.argmax(u)])
        assert u.max() <= bound, (u.max(), a[np.argmax(u)])
    y = _run(mechs, 0, np.array([np.nan, np.inf, -np.inf, -708.5, 710.0, 0.0, -0.0]))
    assert np.isnan(y[0]) and y[1] == np.inf and y[4] == np.inf and (y[2:4] == 0.0).all() and (y[5:] == 1.0).all()


def test_log(mechs):
    rng = np.random.default_rng(3)
    edges = np.arange(96, 193) / 128.0            # the table's intervals and the seams between them
    seams = (np.arange(96, 193) + 0.5) / 128.0
    x = np.concatenate([10.0 ** rng.uniform(-307, 308, 60000), rng.uniform(200.0, 6000.0, 40000),
                        rng.uniform(0.5, 2.0, 60000), 1.0 + _near(rng, 20000, 1e-16, 0.01),
                        *(q * (1.0 + d) * 2.0 ** e for q in (edges, seams) for d in (-2e-16, 0.0, 2e-16)
                          for e in (-1, 0, 1, 12))])
    u = np.where(x == 1.0, 0.0, _ulp(_run(mechs, 3, x), np.where(x == 1.0, LD(1), np.log(x.astype(LD)))))
    print("log worst", u.max(), "at", x[np.argmax(u)])
    assert u.max() <= 1.5, (u.max(), x[np.argmax(u)])
    sub = np.array([5e-324, 1e-310, 2.2250738585072014e-308, 1.7976931348623157e308])
    assert _ulp(_run(mechs, 3, sub), np.log(sub.astype(LD))).max() <= 1.5
    y = _run(mechs, 3, np.array([1.0, 0.0, -0.0, -1.0, np.inf, np.nan]))
    assert y[0] == 0.0 and (y[1:3] == -np.inf).all() and np.isnan(y[3]) and y[4] == np.inf and np.isnan(y[5])
