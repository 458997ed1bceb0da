"""Direct integration gives a cell the same bits whether one warp integrates it or a team of warps:
every sum runs in the same order in both.  Calls on both sides of the team forms' limits (one cell; a
round of teams; a few more; many), subsets through an index list, and cells that are refused before
their first step.  The learned step's fallback, whose cell count only the device knows, takes either form.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2402_18858_gb300 import workload as w  # noqa: E402


def _setup(kind, tmp_path, n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2402_18858_gb300 import build, chem as lc
    build.build()
    m = w.make_mechanism(kind, {"h2_9": 0, "c_30": 1, "c_53": 5}[kind])
    path = str(tmp_path / "m.mech")
    w.write_mechanism(m, path)
    st = w.make_states(m, n, 31)
    st.T[3] = -5.0
    st.Y[1, 7] = np.nan
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")  # noqa: E731
    return lc, lc.chem_load_mech(path), dev, dev(st.T), dev(st.p), dev(st.Y)


@pytest.mark.parametrize("kind", ["h2_9", "c_30", "c_53"])
def test_small_and_large_calls_agree(kind, tmp_path):
    N = 2600
    lc, gm, dev, T0, p, Y0 = _setup(kind, tmp_path, N)
    queue = torch.empty(256, dtype=torch.uint8, device="cuda")

    def run(idx):
        T, Y = T0.clone(), Y0.clone()
        status = torch.full((idx.numel(),), -1, dtype=torch.int32, device="cuda")
        stats = torch.full((4, idx.numel()), -1, dtype=torch.int32, device="cuda")
        lc.chem_step_di(gm, 1e-5, T, p, Y, status, idx=idx, stats=stats, workspace=queue, rtol=1e-6, atol_Y=1e-12)
        return T, Y, status, stats

    T, Y, status, stats = run(torch.arange(N, dtype=torch.int32, device="cuda"))
    assert status[3] != 0 and status[7] != 0 and int((status == 0).sum()) >= N - 2
    rng = np.random.default_rng(4)
    for n in (1, 5, 152, 300, 456, 457, 1000):
        perm = rng.permutation(N)[:n].astype(np.int32)
        if n >= 5:
            perm = np.unique(np.concatenate([perm, np.array([3, 7], np.int32)]))[:n]
        idx = dev(perm)
        li = idx.long()
        Tn, Yn, sn, kn = run(idx)
        assert torch.equal(sn, status[li])
        a, b = Tn[li].view(torch.int64), T[li].view(torch.int64)
        assert torch.equal(a, b), (n, int((a != b).sum()))
        a, b = Yn[:, li].contiguous().view(torch.int64), Y[:, li].contiguous().view(torch.int64)
        assert torch.equal(a, b), (n, int((a != b).sum()))
        assert torch.equal(kn, stats[:, li])


@pytest.mark.parametrize("kind", ["h2_9", "c_30", "c_53"])
@pytest.mark.parametrize("n", [1, 400, 2000])
def test_fallback_equals_direct_integration(kind, n, tmp_path):
    """All cells fall back (no temperature change is allowed): a few, about a round of teams, many."""
    lc, gm, dev, T0, p, Y0 = _setup(kind, tmp_path, 2000)
    ann = lc.chem_ann_create(gm, [16], seed=1)
    idx = torch.arange(100 if n < 2000 else 0, 100 + n if n < 2000 else n, dtype=torch.int32, device="cuda")
    ws = torch.empty(lc.chem_ann_workspace_bytes(ann, n), dtype=torch.uint8, device="cuda")
    queue = torch.empty(256, dtype=torch.uint8, device="cuda")
    T, Y = T0.clone(), Y0.clone()
    status = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    lc.chem_step_ann(gm, ann, 5e-6, T, p, Y, status, ws, idx=idx, T_min=9998.0, T_max=9999.0, di_rtol=1e-6, di_atol_Y=1e-12)
    Td, Yd = T0.clone(), Y0.clone()
    sd = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    lc.chem_step_di(gm, 5e-6, Td, p, Yd, sd, idx=idx, workspace=queue, rtol=1e-6, atol_Y=1e-12)
    assert torch.equal(status == 5, sd == 0)
    assert torch.equal(T.view(torch.int64), Td.view(torch.int64))
    assert torch.equal(Y.view(torch.int64), Yd.view(torch.int64))
