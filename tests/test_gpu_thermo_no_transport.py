"""Properties without transport outputs: c_p, h and T from h are the same FP64 sums in both precision modes,
so the modes give the same bits (also for cells that are not finite), whatever outputs are asked for, and
agree with those of a call with transport outputs to 1e-12 (another summation order).  Species counts with
an unrolled kernel and without, calls of one cell, of a block and a remainder, of many.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2402_18858_gb300 import workload as w  # noqa: E402


@pytest.mark.parametrize("K", [9, 22, 30, 41, 53])
@pytest.mark.parametrize("n", [1, 257, 20_000])
def test_modes_agree(K, n, tmp_path, monkeypatch):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2402_18858_gb300 import build, chem as lc
    build.build()
    kind = {9: "h2_9", 30: "c_30", 53: "c_53"}.get(K, "sub")
    if kind == "sub":
        species = [s for s in w._SP53 if s != "N2"][:K - 1] + ["N2"]
        monkeypatch.setitem(w.MECH_KINDS, kind, (species, ["C", "H", "O", "N"], "CH4", 3 * K, 3, 3))
    m = w.make_mechanism(kind, 5)
    path = str(tmp_path / "m.mech")
    w.write_mechanism(m, path)
    gm = lc.chem_load_mech(path)
    st = w.make_states(m, n, 11)
    if n > 1:
        st.Y[0, n // 2] = np.nan
        st.T[n - 1] = np.inf
    T, Y = (torch.as_tensor(np.ascontiguousarray(a), device="cuda") for a in (st.T, st.Y))
    new = lambda: torch.full((n,), -1.0, dtype=torch.float64, device="cuda")  # noqa: E731

    def run(mixed, **names):
        o = {k: new() for k in names}
        lc.thermo_props(gm, T, Y, mixed_precision=mixed, **o)
        return o

    both = [run(mixed, cp=1, h=1) for mixed in (False, True)]
    alone = {**run(False, cp=1), **run(False, h=1)}
    full = run(False, cp=1, h=1, mu=1, kappa=1)
    ok = torch.isfinite(full["cp"])
    assert int(ok.sum()) == n - (2 if n > 1 else 0)
    for q in ("cp", "h"):
        assert torch.equal(both[0][q].view(torch.int64), both[1][q].view(torch.int64))
        assert torch.equal(both[0][q].view(torch.int64), alone[q].view(torch.int64))
        # h crosses zero: relative to c_p T
        scale = full["cp"].abs() * (T if q == "h" else 1.0)
        for got in (both[0][q], alone[q]):
            assert ((got - full[q]).abs() <= 1e-12 * (scale + full[q].abs()))[ok].all()
    h_in = torch.where(ok, full["h"], torch.zeros_like(T))
    guess = torch.where(ok, T + 35.0, torch.full_like(T, 1500.0))
    found = []
    for mixed in (False, True):
        T_out, cp = new(), new()
        lc.thermo_props(gm, guess, Y, cp=cp, h_in=h_in, T_out=T_out, mixed_precision=mixed)
        found.append((T_out, cp))
    for a, b in zip(*found):
        assert torch.equal(a.view(torch.int64), b.view(torch.int64))
    # |dT| < 1e-9 K ends the iteration; the error left is quadratic in that, rounding aside
    assert ((found[0][0] - T).abs() <= 1e-9)[ok].all()
