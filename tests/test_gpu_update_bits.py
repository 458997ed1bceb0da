"""The learned step's update gives a cell the same bits in every call, whatever the call's size (its two
forms, a warp per cell and a thread per cell, do the same operations in the same order): temperature, mass
fractions, flags and status are compared as bit patterns between one large call and small ones.  Element
systems of three, four and eight elements, the last with two elements that are multiples of others (a
singular system, which magnifies a difference in a last bit), and cells whose mass fractions are not finite.
The learned step as a whole, whose calls a server cuts and joins by load, likewise.
"""
import dataclasses

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2402_18858_gb300 import workload as w  # noqa: E402

N = 20_000
SMALL = (1, 33, 600, 2100, 5000)
CASES = [("h2_9", 3), ("c_30", 4), ("c_53", 4), ("c_30", 8)]


def _bits(t):
    return t.contiguous().view(torch.int64) if t.dtype == torch.float64 else t


def _setup(kind, elements, tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2402_18858_gb300 import build, chem as lc
    build.build()
    m = w.make_mechanism(kind, {"h2_9": 0, "c_30": 1, "c_53": 5}[kind])
    more = elements - len(m.elements)
    comp = np.pad(m.comp, ((0, 0), (0, more)))
    for q in range(min(more, 2)):
        comp[:, len(m.elements) + q] = (q + 2) * comp[:, q]
    m = dataclasses.replace(m, elements=m.elements + [f"E{q}" for q in range(more)], comp=comp)
    path = str(tmp_path / "m.mech")
    w.write_mechanism(m, path)
    gm = lc.chem_load_mech(path)
    ann = lc.chem_ann_create(gm, [16], seed=1)
    norm = lc.chem_ann_get_norm(ann)
    norm[4 * ann.n_in + m.n_species:] = 0.02
    lc.chem_ann_set_norm(ann, norm)
    return lc, m, gm, ann, w.make_states(m, N, 21)


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


@pytest.mark.parametrize("not_finite", [0.0, 0.25])
@pytest.mark.parametrize("kind,elements", CASES)
def test_update(kind, elements, not_finite, tmp_path):
    lc, m, gm, ann, st = _setup(kind, elements, tmp_path)
    K = m.n_species
    rng = np.random.default_rng(5)
    # cells with one species NaN or infinite; predictions from accepted to far off
    bad = rng.random(N) < not_finite
    st.Y[rng.integers(0, K, N)[bad], np.flatnonzero(bad)] = rng.choice([np.nan, np.inf, -np.inf], int(bad.sum()))
    U = np.zeros((N, ann.n_out_pad), np.float32)
    U[:, :K] = rng.standard_normal((N, K)) * 10.0 ** rng.uniform(-3, 1.0, (N, 1))
    T0, Y0, p, Ud = _dev(st.T), _dev(st.Y), _dev(st.p), _dev(U)

    def run(idx):
        T, Y, n = T0.clone(), Y0.clone(), idx.numel()
        fl = torch.zeros(n, dtype=torch.int32, device="cuda")
        status = torch.full((n,), -1, dtype=torch.int32, device="cuda")
        lc.chem_ann_update(ann, T, p, Y, Ud[idx.long()].contiguous(), fl, status, idx=idx, dT_max=300.0)
        return T, Y, fl, status

    T, Y, fl, status = run(torch.arange(N, dtype=torch.int32, device="cuda"))
    assert {0, 4} <= set(fl.cpu().tolist())
    order = rng.permutation(N).astype(np.int32)
    for n in SMALL:
        idx = _dev(order[:n])
        at = idx.long()
        Ts, Ys, fs, ss = run(idx)
        assert torch.equal(fs, fl[at]) and torch.equal(ss, status[at]), (n, int((fs != fl[at]).sum()))
        assert torch.equal(_bits(Ts[at]), _bits(T[at])), n
        differ = _bits(Ys[:, at]) != _bits(Y[:, at])
        assert not differ.any(), (n, int(differ.sum()))


@pytest.mark.parametrize("kind,elements", CASES[:3])
def test_learned_step(kind, elements, tmp_path):
    lc, m, gm, ann, st = _setup(kind, elements, tmp_path)
    T0, Y0, p = _dev(st.T), _dev(st.Y), _dev(st.p)
    noise = torch.randn(Y0.shape, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    lc.chem_ann_fit_norm(ann, T0, p, Y0, Y0 * (1.0 + 1e-4 * noise))

    def run(idx):
        T, Y, n = T0.clone(), Y0.clone(), idx.numel()
        status = torch.full((n,), -1, dtype=torch.int32, device="cuda")
        ws = torch.empty(lc.chem_ann_workspace_bytes(ann, n), dtype=torch.uint8, device="cuda")
        lc.chem_step_ann(gm, ann, 1e-7, T, p, Y, status, ws, idx=idx, T_min=200.0, T_max=6000.0, no_fallback=True)
        return T, Y, status

    T, Y, status = run(torch.arange(N, dtype=torch.int32, device="cuda"))
    assert int((status == 0).sum()) > N // 100
    order = np.random.default_rng(6).permutation(N).astype(np.int32)
    for n in SMALL:
        idx = _dev(order[:n])
        at = idx.long()
        Ts, Ys, ss = run(idx)
        assert torch.equal(ss, status[at]) and torch.equal(_bits(Ts[at]), _bits(T[at]))
        assert torch.equal(_bits(Ys[:, at]), _bits(Y[:, at])), n
