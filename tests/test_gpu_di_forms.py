"""Direct integration with the number of warps per cell asked for: one warp, a team of two (above 32
unknowns) and a team of four give every cell the same bits and the same step counters, up to and above 32
unknowns.  Mechanisms that have no teams (three partners on a side of a reaction) run one warp per cell,
also above 32 unknowns, and agree with the oracle.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2402_18858_gb300 import workload as w  # noqa: E402


def _mechanism(kind, monkeypatch):
    if kind == "c_36":
        species = w._SP30[:-1] + w._SP53_EXTRA[:6] + ["N2"]
        monkeypatch.setitem(w.MECH_KINDS, kind, (species, ["C", "H", "O", "N"], "CH4", 216, 7, 9))
    return w.make_mechanism(kind, {"h2_9": 0, "c_30": 1, "c_36": 7, "c_53": 5}[kind])


def _load(m, tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2402_18858_gb300 import build, chem as lc
    build.build()
    path = str(tmp_path / "m.mech")
    w.write_mechanism(m, path)
    return lc, lc.chem_load_mech(path), path


def _run(lc, gm, st, call, **kw):
    T, p, Y = (torch.as_tensor(np.ascontiguousarray(a), device="cuda") for a in (st.T, st.p, st.Y))
    n = T.numel()
    status = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    stats = torch.full((4, n), -1, dtype=torch.int32, device="cuda")
    ws = torch.empty(lc.chem_workspace_bytes(gm, n), dtype=torch.uint8, device="cuda")
    call(T, p, Y, status, workspace=ws, stats=stats, **kw)
    return [T.view(torch.int64), Y.view(torch.int64), status, stats]


@pytest.mark.parametrize("kind,forms", [("c_30", (4,)), ("c_36", (2, 4)), ("c_53", (2, 4))])
@pytest.mark.parametrize("n", [3, 700])
def test_forms_agree(kind, forms, n, tmp_path, monkeypatch):
    m = _mechanism(kind, monkeypatch)
    lc, gm, _ = _load(m, tmp_path)
    st = w.make_states(m, n, 31)
    st.T[1] = -5.0      # refused before its first step

    def form(k):
        return _run(lc, gm, st, lambda *a, **kw: lc.chem_selftest_di_form(gm, k, 1e-5, *a, **kw), rtol=1e-6,
                    atol_Y=1e-12)

    one = form(1)
    assert one[2][1] != 0 and int((one[2] == 0).sum()) >= 0.3 * n
    for k in forms:
        for a, b in zip(one, form(k)):
            assert torch.equal(a, b), (k, int((a != b).sum()))
    for a, b in zip(one, _run(lc, gm, st, lambda *a, **kw: lc.chem_step_di(gm, 1e-5, *a, **kw), rtol=1e-6, atol_Y=1e-12)):
        assert torch.equal(a, b)


@pytest.mark.parametrize("n", [1, 400, 900, 2000])
def test_fallback(n, tmp_path, monkeypatch):
    """The learned step's fallback, whose count only the device knows, in a mechanism where each range of
    counts has its own form: n of 2,000 cells are too hot for the learned step."""
    m = _mechanism("c_36", monkeypatch)
    lc, gm, _ = _load(m, tmp_path)
    N = 2000
    st = w.make_states(m, N, 31)
    ann = lc.chem_ann_create(gm, [16], seed=1)
    T, p, Y = (torch.as_tensor(np.ascontiguousarray(a), device="cuda") for a in (st.T, st.p, st.Y))
    Yd = Y.clone()
    status, sd = (torch.full((N,), -1, dtype=torch.int32, device="cuda") for _ in range(2))
    ws = torch.empty(lc.chem_ann_workspace_bytes(ann, N), dtype=torch.uint8, device="cuda")
    ref = torch.empty(lc.chem_workspace_bytes(gm, N), dtype=torch.uint8, device="cuda")
    norm = lc.chem_ann_get_norm(ann)
    norm[4 * ann.n_in + m.n_species:] = 1e-12     # no change predicted: cells are accepted by their temperature
    lc.chem_ann_set_norm(ann, norm)
    flagged = torch.arange(N, device="cuda") < n
    T = torch.where(flagged, T + 1000.0, torch.full_like(T, 1000.0))
    Td = T.clone()
    lc.chem_step_ann(gm, ann, 1e-9, T, p, Y, status, ws, T_max=1100.0, elem_tol=1e9, di_rtol=1e-6,
                     di_atol_Y=1e-12)
    lc.chem_selftest_di_form(gm, 1, 1e-9, Td, p, Yd, sd, ref, rtol=1e-6, atol_Y=1e-12)
    assert torch.equal(status != 0, flagged)
    assert torch.equal(status[flagged] == 5, sd[flagged] == 0)
    assert torch.equal(T.view(torch.int64)[flagged], Td.view(torch.int64)[flagged])
    assert torch.equal(Y[:, flagged].contiguous().view(torch.int64), Yd[:, flagged].contiguous().view(torch.int64))


@pytest.mark.parametrize("kind", ["h2_9", "c_30", "c_36"])
def test_without_teams(kind, tmp_path, monkeypatch):
    from oracle import Oracle
    m = _mechanism(kind, monkeypatch)
    i = m.index
    m.reactions.append(w.Reaction(0, [i("H"), i("O2"), i("H2O")], [i("HO2"), i("H2O")], 1e-2, 0.1, 1e4))
    lc, gm, path = _load(m, tmp_path)
    n, dt = 24, 1e-6
    st = w.make_states(m, n, 7)
    for k in (2, 4):
        with pytest.raises(lc.ChemError):
            _run(lc, gm, st, lambda *a, **kw: lc.chem_selftest_di_form(gm, k, dt, *a, **kw))
    got = _run(lc, gm, st, lambda *a, **kw: lc.chem_step_di(gm, dt, *a, **kw))
    T, Y = (t.view(torch.float64).cpu().numpy() for t in got[:2])
    To, Yo, so, _ = Oracle(path).integrate_batch(st.T, st.p, st.Y, dt)
    # (a random mechanism can be too stiff for the step limit of either side in single cells)
    ok = (got[2].cpu().numpy() == 0) & (so == 0)
    assert ok.mean() > 0.8
    # the parity criterion of the integration: 1e-6 on T and on every fraction above 1e-10
    assert (np.abs(T - To) <= 1e-6 * To)[ok].all()
    assert (np.abs(Y - Yo) <= 1e-6 * Yo)[(Yo > 1e-10) & ok].all()
