"""Arrays that kernels move 16 (or count 4) bytes at a time are refused on the host when they start elsewhere:
the features, and the workspaces of the learned step, the network and the direct integration.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2402_18858_gb300 import workload as w  # noqa: E402


def test_misaligned_arrays_are_refused(mechs):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2402_18858_gb300 import build, chem as lc
    build.build()
    m, path = mechs["h2_9"]
    gm = lc.chem_load_mech(path)
    ann = lc.chem_ann_create(gm, [16], seed=1)
    n = 40
    st = w.make_states(m, n, 3)
    T, p, Y = (torch.as_tensor(np.ascontiguousarray(a), device="cuda") for a in (st.T, st.p, st.Y))
    status = torch.zeros(n, dtype=torch.int32, device="cuda")
    X = torch.zeros(n * 64 + 1, dtype=torch.bfloat16, device="cuda")
    U = torch.zeros((n, ann.n_out_pad), device="cuda")
    ws = torch.zeros(lc.chem_ann_workspace_bytes(ann, n) + 8, dtype=torch.uint8, device="cuda")
    wd = torch.zeros(lc.chem_workspace_bytes(gm, n) + 2, dtype=torch.uint8, device="cuda")
    with pytest.raises(lc.ChemError):
        lc.chem_ann_features(ann, T, p, Y, X[1:].view(n, 64))
    with pytest.raises(lc.ChemError):
        lc.chem_ann_forward(ann, X[:-1].view(n, 64), U, ws[8:])
    with pytest.raises(lc.ChemError):
        lc.chem_step_ann(gm, ann, 1e-6, T, p, Y, status, ws[8:])
    with pytest.raises(lc.ChemError):
        lc.chem_step_di(gm, 1e-6, T, p, Y, status, workspace=wd[2:])
    lc.chem_ann_features(ann, T, p, Y, X[:-1].view(n, 64))
    lc.chem_ann_forward(ann, X[:-1].view(n, 64), U, ws[:-8])
    lc.chem_step_di(gm, 1e-6, T, p, Y, status, workspace=wd[:-2])
    torch.cuda.synchronize()
    assert lc.chem_ann_error(ann) == 0
