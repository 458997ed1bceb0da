"""Hidden-layer epilogues (bias + GELU; times GELU') on widths whose last chunk has 8, 16 or 24 of 32
columns, for the short-K kernel, single CTAs and CTA pairs, against FP64.  The tolerance: products of
BF16 in FP32 (1e-5 of the sum of magnitudes, through the slope), one BF16 rounding (2^-8), and the
approximate erf (1e-6 of the largest value).
"""
import math

import numpy as np
import pytest
from scipy.special import erf

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPES = [(130, 8, 64), (257, 24, 64), (129, 2000, 64), (300, 40, 72), (33, 16, 200), (300, 104, 304),
          (130, 504, 1000), (515, 1000, 520)]


@pytest.mark.parametrize("M,N,K", SHAPES)
@pytest.mark.parametrize("epi", [0, 2])
def test_last_chunk(M, N, K, epi):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2402_18858_gb300 import build, chem as lc
    build.build()
    rng = np.random.default_rng(M + 3 * N + K + epi)
    bf = lambda shape, s=1.0: torch.as_tensor(rng.standard_normal(shape) * s, dtype=torch.float32).to(torch.bfloat16)  # noqa: E731
    A, B, z = bf((M, K)), bf((N, K), 1.0 / math.sqrt(K)), bf((M, N))
    bias = torch.as_tensor(rng.standard_normal(N) * 0.1, dtype=torch.float32)
    guard = 64      # rows after the result, which the kernel must leave alone
    buf = torch.full((M + guard, N), 7.0, dtype=torch.bfloat16, device="cuda")
    err = lc.chem_selftest_gemm(epi, A.cuda(), B.cuda(), buf[:M], bias=bias.cuda() if epi == 0 else None,
                                z=z.cuda() if epi == 2 else None)
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    assert bool((buf[M:] == 7.0).all())
    a, b = A.double().numpy(), B.double().numpy()
    acc, bound = a @ b.T, 1e-5 * (np.abs(a) @ np.abs(b).T)
    x = acc + bias.double().numpy()[None, :] if epi == 0 else z.double().numpy()
    phi = 0.5 * (1.0 + erf(x / math.sqrt(2.0)))
    slope = phi + x * np.exp(-0.5 * x * x) / math.sqrt(2 * math.pi)
    ref = x * phi if epi == 0 else acc * slope
    tol = np.abs(slope) * bound + 2.0 ** -8 * np.abs(ref) + 1e-6 * np.abs(ref).max()
    got = buf[:M].double().cpu().numpy()
    assert (np.abs(got - ref) <= tol).all(), np.abs(got - ref).max()
