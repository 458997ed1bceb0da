"""Properties over species counts and inputs at the edges of the kernels' layouts: every
instantiation's first, last and next species count, cells of both NASA-7 ranges side by side, absent
and slightly negative species, one-species cells, T from h across the range boundary, and inputs
that are not finite or far outside the fixed-point form's exponents.

Reference: the textbook formulas in FP64 numpy.  FP64 mode: 1e-12 relative (about 30 species-sum
roundings of 1e-16 and the exponential of a fit of magnitude up to 30); the FP32 transport sums of
the mixed mode: 2e-5.
"""
import dataclasses

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2402_18858_gb300 import workload as w  # noqa: E402

R = 8.314462618


def _mech(K, tmp_path):
    """K species drawn from the 53-species set (names made unique past 53), one exchange reaction."""
    m = w.make_mechanism("c_53", 5)
    pick = np.arange(K) % m.n_species
    m = dataclasses.replace(m, species=[f"S{i}" for i in range(K)], comp=m.comp[pick], W=m.W[pick],
                            nasa_low=m.nasa_low[pick], nasa_high=m.nasa_high[pick], mu_fit=m.mu_fit[pick],
                            lam_fit=m.lam_fit[pick], reactions=[w.Reaction(0, [0], [0], 1.0, 0.0, 0.0)])
    path = str(tmp_path / f"k{K}.mech")
    w.write_mechanism(m, path)
    return m, path


def _cp_h(m, T, Y):
    a = np.where((T >= m.T_mid)[None, None, :], m.nasa_high[:, :, None], m.nasa_low[:, :, None])
    cp = sum(a[:, i] * T ** i for i in range(5))
    h = sum(a[:, i] * T ** (i + 1) / (i + 1) for i in range(5)) + a[:, 5]
    yw = Y / m.W[:, None]
    return R * (yw * cp).sum(axis=0), R * (yw * h).sum(axis=0)


def _reference(m, T, Y):
    cp, h = _cp_h(m, T, Y)
    X = Y / m.W[:, None]
    X = X / X.sum(axis=0)
    L = np.log(T)
    mu = np.exp(sum(m.mu_fit[:, i:i + 1] * L ** i for i in range(4)))
    lam = np.exp(sum(m.lam_fit[:, i:i + 1] * L ** i for i in range(4)))
    mix = np.zeros_like(T)
    for k in range(m.n_species):
        f = (1 + np.sqrt(mu[k] / mu) * ((m.W / m.W[k]) ** 0.25)[:, None]) ** 2 / np.sqrt(8 * (1 + m.W[k] / m.W))[:, None]
        mix += X[k] * mu[k] / (X * f).sum(axis=0)
    return cp, h, mix, 0.5 * ((X * lam).sum(axis=0) + 1 / (X / lam).sum(axis=0))


def _states(K, n, rng):
    T = rng.uniform(300.0, 2800.0, n)
    Y = 10.0 ** rng.uniform(-9, 0, (K, n))
    Y[rng.random((K, n)) < 0.2] = 0.0
    Y[0] += 1e-3
    Y /= Y.sum(axis=0)
    Y[:, 0] = 0.0
    Y[K - 1, 0] = 1.0                       # one species
    if K > 1:
        Y[0, 1] = -1e-12                    # undershoot of a transport scheme
    return T, Y


@pytest.mark.parametrize("K", [1, 2, 9, 10, 16, 17, 24, 25, 30, 31, 40, 41, 53, 54, 55, 62, 63])
def test_properties_at_layout_edges(K, tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2402_18858_gb300 import build, chem as lc
    build.build()
    m, path = _mech(K, tmp_path)
    gm = lc.chem_load_mech(path)
    rng = np.random.default_rng(K)
    n, ld = 77, 83
    T, Y = _states(K, ld, rng)
    ref = _reference(m, T, Y)
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")  # noqa: E731
    Td, Yd = dev(T), dev(Y)
    for mixed, tol in ((False, 1e-12), (True, 2e-5)):
        out = [torch.full((ld,), -7.0, dtype=torch.float64, device="cuda") for _ in range(4)]
        lc.thermo_props(gm, Td, Yd, *out, mixed_precision=mixed, n=n)
        for q, (o, r) in enumerate(zip(out, ref)):
            o = o.cpu().numpy()
            scale = np.abs(r[:n]) + (1e-3 * np.abs(ref[0] * T)[:n] if q == 1 else 0.0)   # h passes through zero
            assert (np.abs(o[:n] - r[:n]) <= (1e-12 if q < 2 else tol) * scale).all(), (mixed, q)
            assert (o[n:] == -7.0).all()
        # one output at a time gives the same bits
        mu = torch.empty(ld, dtype=torch.float64, device="cuda")
        lc.thermo_props(gm, Td, Yd, mu=mu, mixed_precision=mixed, n=n)
        assert torch.equal(mu[:n], out[2][:n])
        # T from h: guesses on the other side of the range boundary among them, T written in place
        Tg = dev(np.where(np.arange(ld) % 3 == 0, 2200.0 - 0.5 * T, T + 40.0))
        cp = torch.empty(ld, dtype=torch.float64, device="cuda")
        lc.thermo_props(gm, Tg, Yd, cp=cp, h_in=dev(ref[1]), T_out=Tg, mixed_precision=mixed, n=n)
        assert (np.abs(Tg.cpu().numpy()[:n] - T[:n]) <= 1e-8).all()
        assert (np.abs(cp.cpu().numpy()[:n] - ref[0][:n]) <= 1e-10 * ref[0][:n]).all()


@pytest.mark.parametrize("K", [9, 30, 53])
def test_properties_of_extreme_inputs(K, tmp_path):
    """Cells the fixed-point form does not take: scaled far up or down (the mixture's transport does
    not depend on the scale, c_p and h are linear in it), and NaN, infinite or zero inputs, whose
    outputs are not finite; their neighbours keep their values."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2402_18858_gb300 import build, chem as lc
    build.build()
    m, path = _mech(K, tmp_path)
    gm = lc.chem_load_mech(path)
    n = 40
    T, Y = _states(K, n, np.random.default_rng(100 + K))
    ref = _reference(m, T, Y)
    s = np.ones(n)
    s[[3, 4]] = 1e150, 1e-150
    Y2, T2 = Y * s, T.copy()
    Y2[1, 10] = np.nan
    Y2[1, 11] = np.inf
    Y2[:, 12] = 0.0
    T2[13] = np.nan
    out = [torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(4)]
    lc.thermo_props(gm, torch.as_tensor(T2, device="cuda"), torch.as_tensor(Y2, device="cuda"), *out)
    cp, h, mu, kap = (o.cpu().numpy() for o in out)
    ok = np.ones(n, bool)
    ok[10:14] = False
    for o, r in ((cp, ref[0] * s), (mu, ref[2]), (kap, ref[3])):
        assert (np.abs(o - r)[ok] <= 1e-12 * np.abs(r)[ok]).all()
    assert (np.abs(h - ref[1] * s)[ok] <= 1e-12 * (np.abs(ref[1]) + 1e-3 * np.abs(ref[0] * T))[ok] * s[ok]).all()
    for o in (mu, kap):
        assert not np.isfinite(o[10:14]).any()
    assert not np.isfinite(cp[[10, 11, 13]]).any() and cp[12] == 0.0
