"""The learned step's update has two forms, a warp per cell for calls with few cells and a thread per
cell for many.  Every cell gives the same result in a small call and in a large one: the temperature,
flags and status bit for bit (all FP32 sums run in the same order), the mass fractions within 1e-12
(the FP64 element projection; its E x E system is ill-conditioned by up to about 1e3).  Three, four and
eight elements (element counts of the instantiations, the last with elements that no species has),
predictions of every flag, non-finite ones among them, and an index list.
"""
import dataclasses

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2402_18858_gb300 import workload as w  # noqa: E402


@pytest.mark.parametrize("kind,elements", [("h2_9", 3), ("c_30", 4), ("c_53", 4), ("c_30", 8)])
def test_small_and_large_calls_agree(kind, elements, tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2402_18858_gb300 import build, chem as lc
    build.build()
    m = w.make_mechanism(kind, {"h2_9": 0, "c_30": 1, "c_53": 5}[kind])
    more = elements - len(m.elements)
    m = dataclasses.replace(m, elements=m.elements + [f"E{q}" for q in range(more)],
                            comp=np.pad(m.comp, ((0, 0), (0, more))))
    path = str(tmp_path / "m.mech")
    w.write_mechanism(m, path)
    gm = lc.chem_load_mech(path)
    K, N = m.n_species, 20_000
    ann = lc.chem_ann_create(gm, [16], seed=1)
    norm = lc.chem_ann_get_norm(ann)
    norm[4 * ann.n_in + K:] = 0.02
    lc.chem_ann_set_norm(ann, norm)
    st = w.make_states(m, N, 21)
    rng = np.random.default_rng(5)
    U = np.zeros((N, ann.n_out_pad), np.float32)
    U[:, :K] = rng.standard_normal((N, K)) * 10.0 ** rng.uniform(-3, 1.5, (N, 1))
    U[5, 0], U[6, 1], U[7, :K] = np.nan, np.inf, -1e6
    flags0 = (rng.random(N) < 0.05).astype(np.int32)
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")  # noqa: E731
    p, Ud = dev(st.p), dev(U)

    def run(idx):
        n = idx.numel()
        T, Y = dev(st.T), dev(st.Y)
        fl, status = dev(flags0)[idx.long()].contiguous(), torch.full((n,), -1, dtype=torch.int32, device="cuda")
        lc.chem_ann_update(ann, T, p, Y, Ud[idx.long()].contiguous(), fl, status, idx=idx, dT_max=300.0)
        return T, Y, fl, status

    everything = torch.arange(N, dtype=torch.int32, device="cuda")
    T, Y, fl, status = run(everything)
    seen = set(fl.cpu().tolist())
    assert {0, 1, 2, 4} <= seen, seen
    for n in (1, 5, 33, 3001):
        idx = dev(rng.permutation(N)[:n].astype(np.int32))
        if n == 33:
            idx[:3] = dev(np.array([5, 6, 7], np.int32))
        Ts, Ys, fs, ss = run(idx)
        at = idx.long()
        assert torch.equal(fs, fl[at]) and torch.equal(ss, status[at])
        assert torch.equal(Ts[at], T[at])
        assert ((Ys[:, at] - Y[:, at]).abs() <= 1e-12 * Y[:, at].abs() + 1e-300).all()
        rest = torch.ones(N, dtype=torch.bool, device="cuda")
        rest[at] = False
        assert torch.equal(Ts[rest], dev(st.T)[rest]) and torch.equal(Ys[:, rest], dev(st.Y)[:, rest])
