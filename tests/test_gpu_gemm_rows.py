"""GEMM results whose rows, biases or first element do not start on 16 bytes: widths from 32 columns up
that are no multiple of 8 (BF16 results) or 4 (FP32 results), a result and biases at odd offsets, all four
epilogues, the short-K kernel, single CTAs and CTA pairs, against FP64; and the network's output written
to an array that starts 4 bytes off.  The elements around the result stay as they were.  The tolerances are
those of the aligned widths: products of BF16 in FP32 (1e-5 of the sum of magnitudes, through the slope),
one BF16 rounding (2^-8) and the approximate erf (1e-6 of the largest value).
"""
import math

import numpy as np
import pytest
from scipy.special import erf

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2402_18858_gb300 import workload as w  # noqa: E402


@pytest.mark.parametrize("M,N,K", [(130, 33, 64), (257, 36, 128), (129, 100, 72), (300, 130, 200), (515, 260, 520),
                                   (33, 61, 304), (130, 64, 64), (300, 160, 304)])
@pytest.mark.parametrize("epi", [0, 1, 2, 3])
@pytest.mark.parametrize("off", [0, 1])
def test_rows_off_16_bytes(M, N, K, epi, off):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2402_18858_gb300 import build, chem as lc
    build.build()
    rng = np.random.default_rng(M + 3 * N + K + epi)
    bf = lambda shape, s=1.0: torch.as_tensor(rng.standard_normal(shape) * s, dtype=torch.float32).to(torch.bfloat16)  # noqa: E731
    A, B, z = bf((M, K)), bf((N, K), 1.0 / math.sqrt(K)), bf((M, N))
    bias = torch.as_tensor(rng.standard_normal(N) * 0.1, dtype=torch.float32)

    def at(t):      # t on the GPU, `off` elements behind an allocation's start
        b = torch.empty(t.numel() + off, dtype=t.dtype, device="cuda")
        b[off:] = t.cuda().flatten()
        return b[off:].view(t.shape)

    buf = torch.full((off + M * N + 64,), 7.0, dtype=torch.bfloat16 if epi in (0, 2) else torch.float32, device="cuda")
    out = buf[off:off + M * N].view(M, N)
    err = lc.chem_selftest_gemm(epi, A.cuda(), B.cuda(), out, bias=at(bias) if epi < 2 else None,
                                z=at(z) if epi == 2 else None)
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    assert bool((buf[:off] == 7.0).all()) and bool((buf[off + M * N:] == 7.0).all())
    a, b = A.double().numpy(), B.double().numpy()
    acc, bound = a @ b.T, 1e-5 * (np.abs(a) @ np.abs(b).T) + 1e-30
    got = out.double().cpu().numpy()
    if epi in (1, 3):
        ref = acc + bias.double().numpy()[None, :] if epi == 1 else acc
        assert (np.abs(got - ref) <= bound + 1e-7 * np.abs(ref)).all()
        return
    x = acc + bias.double().numpy()[None, :] if epi == 0 else z.double().numpy()
    phi = 0.5 * (1.0 + erf(x / math.sqrt(2.0)))
    slope = phi + x * np.exp(-0.5 * x * x) / math.sqrt(2 * math.pi)
    ref = x * phi if epi == 0 else acc * slope
    tol = np.abs(slope) * bound + 2.0 ** -8 * np.abs(ref) + 1e-6 * np.abs(ref).max()
    assert (np.abs(got - ref) <= tol).all(), np.abs(got - ref).max()


@pytest.mark.parametrize("kind,per_species", [("h2_9", True), ("c_30", False), ("c_53", False)])
def test_forward_output_off_16_bytes(mechs, kind, per_species):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2402_18858_gb300 import build, chem as lc
    build.build()
    gm = lc.chem_load_mech(mechs[kind][1])
    ann = (lc.chem_ann_create_per_species if per_species else lc.chem_ann_create)(gm, [48, 24], seed=3)
    n = 700
    X = torch.randn((n, 64), device="cuda").bfloat16()
    ws = torch.empty(lc.chem_ann_workspace_bytes(ann, n), dtype=torch.uint8, device="cuda")
    whole = torch.zeros(n * ann.n_out_pad, device="cuda")
    lc.chem_ann_forward(ann, X, whole.view(n, ann.n_out_pad), ws)
    off = torch.zeros(n * ann.n_out_pad + 2, device="cuda")
    lc.chem_ann_forward(ann, X, off[1:-1].view(n, ann.n_out_pad), ws)
    assert lc.chem_ann_error(ann) == 0
    assert torch.equal(off[1:-1], whole) and float(off[0]) == 0.0 and float(off[-1]) == 0.0
