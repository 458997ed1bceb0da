"""The PaSR source for every number of species chunks and for whole and ragged last chunks (a chunk is 10
species), calls of one cell, of a block and a remainder, and of more cells than one round of blocks, rows
longer than the call: against the FP64 oracle, at the bound of the other PaSR tests (2e-6: the mixing time
and the search for the slowest formation are FP32).  Rows past the call's cells stay as they were.
"""
import dataclasses

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.pasr import pasr_source  # noqa: E402
from paper_2402_18858_gb300 import workload as w  # noqa: E402

TOL = 2e-6


@pytest.mark.parametrize("K", [1, 9, 10, 11, 19, 20, 21, 31, 40, 44, 50, 57, 60, 63])
@pytest.mark.parametrize("n", [1, 131, 90_001])
def test_sizes(K, n, tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2402_18858_gb300 import build, chem as lc
    build.build()
    m = w.make_mechanism("c_53", 5)
    pick = np.arange(K) % m.n_species
    m = dataclasses.replace(m, species=[f"S{i}" for i in range(K)], comp=m.comp[pick], W=m.W[pick],
                            nasa_low=m.nasa_low[pick], nasa_high=m.nasa_high[pick], mu_fit=m.mu_fit[pick],
                            lam_fit=m.lam_fit[pick], reactions=[w.Reaction(0, [0], [0], 1.0, 0.0, 0.0)])
    path = str(tmp_path / "m.mech")
    w.write_mechanism(m, path)
    gm = lc.chem_load_mech(path)
    rng = np.random.default_rng(K + n)
    Y0 = 10.0 ** rng.uniform(-12, 0, (K, n))
    Y1 = Y0 * (1.0 + rng.choice([-1.0, 0.0, 1.0], (K, n)) * 10.0 ** rng.uniform(-12, -1, (K, n)))
    per = [10.0 ** rng.uniform(a, b, n) for a, b in ((-1, 0), (-3, 1), (0, 6), (-5, -3))]
    per[1][rng.random(n) < 0.1] = 0.0
    ld, dt = n + 3, 1e-6
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")  # noqa: E731
    wide = lambda a: dev(np.pad(a, ((0, 0), (0, ld - n)), constant_values=0.25))  # noqa: E731
    om = torch.full((K, ld), 7.0, dtype=torch.float64, device="cuda")
    kap = torch.full((ld,), 7.0, dtype=torch.float64, device="cuda")
    lc.chem_pasr_source(gm, dt, dev(per[0]), wide(Y0), wide(Y1), *(dev(a) for a in per[1:]), om, kap, n=n)
    om, kap = om.cpu().numpy(), kap.cpu().numpy()
    assert (om[:, n:] == 7.0).all() and (kap[n:] == 7.0).all()
    om_o, kap_o = pasr_source(per[0], Y0, Y1, dt, *per[1:])
    assert (np.abs(kap[:n] - kap_o) <= TOL * kap_o + 1e-300).all()
    assert (np.abs(om[:, :n] - om_o) <= TOL * np.abs(om_o) + 1e-300).all()
