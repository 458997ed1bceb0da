"""The PaSR kernel's formed decision, gain > r_min Y(t+dt), at and around equality: it must be the
IEEE FP64 comparison for every gain, also where an FP32 look at the operands cannot tell, for
thresholds and mass fractions inside and outside FP32's range.  A cell with one species at the
threshold and none formed otherwise has kappa = 0, and kappa > 0 when it is formed.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2402_18858_gb300 import workload as w  # noqa: E402


@pytest.mark.parametrize("kind", ["h2_9", "c_30", "c_53"])
@pytest.mark.parametrize("r_min,y_min,scale", [(0.25, 0.0, 1.0), (1e-9, -1.0, 1.0), (0.3, 0.0, 1e-60), (0.0, 0.0, 1.0),
                                               (1e-40, 0.0, 1.0), (0.1, 1e-3, 1e3)])
def test_formed_decision_at_the_threshold(mechs, kind, r_min, y_min, scale):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2402_18858_gb300 import build, chem as lc
    build.build()
    m, path = mechs[kind]
    gm = lc.chem_load_mech(path)
    K, n = m.n_species, 4000
    rng = np.random.default_rng(7)
    y1 = rng.uniform(0.01, 1.0, n) * scale
    rel = rng.choice([0.0, 1.0, -1.0], n) * 10.0 ** rng.uniform(-16, -4, n)
    Y1 = np.full((K, n), 0.5 * scale)
    Y0 = Y1.copy()                                     # every other species at rest
    k = np.arange(n) % K
    Y1[k, np.arange(n)] = y1
    Y0[k, np.arange(n)] = y1 - r_min * y1 * (1.0 + rel)
    d = Y1 - Y0
    formed = ((d > r_min * Y1) & (Y1 >= (1e-10 if y_min < 0 else y_min))).any(axis=0)
    if r_min == 0.25:
        assert 0.2 < formed.mean() < 0.8
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")  # noqa: E731
    om = torch.empty((K, n), dtype=torch.float64, device="cuda")
    kap = torch.empty(n, dtype=torch.float64, device="cuda")
    one = np.ones(n)
    lc.chem_pasr_source(gm, 1e-6, dev(one), dev(Y0), dev(Y1), dev(one), dev(1e4 * one), dev(1e-4 * one), om, kap,
                        y_min=y_min, r_min=r_min)
    kap = kap.cpu().numpy()
    assert ((kap > 0.0) == formed).all()
